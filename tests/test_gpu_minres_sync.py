"""Hand-overs inside the on-chip MINRES forms: repeated solves agree bit for bit
(every sum has a fixed order, so a scalar read before it was written shows as a
difference), and a wait that gives up is reported by every CTA alike."""
import pytest

from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L, kind", [(16, "row"), (16, "id"), (18, "row")])
def test_repeated_one_reduction_solves_identical(L, kind):
    """The one-reduction row form: 40 capped solves (replacement steps among their
    iterations), the same bits each time."""
    hs = need_gpu()
    with hs.Chain(L, inputs.disorder(L, 3.0, 2), sigma=0.1234) as c:
        b = to_dev(inputs.gaussian(c.n, 5))
        first = None
        for _ in range(40):
            x, info = c.minres(b, tol=0.0, kmax=60, precond=kind, allow_not_converged=True)
            assert info["form"] == hs.FORM_SMEM1 and info["iters"] == 60
            first = x if first is None else first
            assert torch.equal(x, first)
