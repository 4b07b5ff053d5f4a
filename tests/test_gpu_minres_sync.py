"""Hand-overs inside the on-chip MINRES forms: repeated solves agree bit for bit
(every sum has a fixed order, so a scalar read before it was written shows as a
difference), and a wait that gives up is reported by every CTA alike."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import hamiltonian
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


@pytest.mark.parametrize("L, cs", [(4, 1), (8, 1), (10, 4), (12, 8), (14, 16)])
def test_cluster_wait_limit(L, cs, monkeypatch):
    """The cluster form with a wait limit of zero polls (HS_BARRIER_LIMIT): every
    CTA gives up at once, the solve reports HS_TIMEOUT in both precisions, and the
    next solve is right (true residual by the oracle's A)."""
    hs = need_gpu()
    monkeypatch.setenv("HS_MINRES_CLUSTER", str(cs))
    hv = inputs.disorder(L, 3.0, L)
    H, diag, st = hamiltonian.build(L, hv)
    sigma = 0.1234
    A = (H - sigma * sp.identity(len(st))).tocsr()
    M = hamiltonian.precond_diag(H, diag, sigma, "row")
    b = inputs.gaussian(len(st), 3)
    with hs.Chain(L, hv, sigma=sigma) as c:
        for _ in range(2):
            with monkeypatch.context() as m:
                m.setenv("HS_BARRIER_LIMIT", "0")
                for solve, rhs in ((c.minres, to_dev(b)), (c.minres_f32, to_dev(b).float())):
                    with pytest.raises(hs.HSError) as e:
                        solve(rhs)
                    assert e.value.status == hs.HS_TIMEOUT
            x, info = c.minres(to_dev(b), tol=1e-12)
            assert info["form"] == hs.FORM_SMEM
            r = b - A @ x.cpu().numpy()
            assert np.sqrt(r @ (r / M)) <= 5e-12 * np.sqrt(b @ (b / M))


def test_cluster_sweep_wait_limit(tmp_path, monkeypatch):
    """The same in a sweep of two lengths: HS_TIMEOUT, and the next one is right."""
    hs = need_gpu()
    monkeypatch.setenv("HS_SWEEP_TUNE", str(tmp_path / "tune.json"))
    Ls = [8, 10, 10, 8]
    fields = [inputs.disorder(L, 3.0, 60 + r) for r, L in enumerate(Ls)]
    with monkeypatch.context() as m:
        m.setenv("HS_BARRIER_LIMIT", "0")
        with pytest.raises(hs.HSError) as e:
            hs.sweep(Ls, fields, 3)
        assert e.value.status == hs.HS_TIMEOUT
    ev, _, _, _, info = hs.sweep(Ls, fields, 3)
    assert info["converged"] == len(Ls)
    for r, (L, h) in enumerate(zip(Ls, fields)):
        w = np.linalg.eigvalsh(hamiltonian.build(L, h)[0].toarray())
        near = w[np.lexsort((w, np.abs(w - 0.5 * (w[0] + w[-1]))))[:3]]
        assert np.abs(ev[r] - near).max() < 1e-10
