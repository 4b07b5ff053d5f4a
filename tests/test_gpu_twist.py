"""GPU parity of the twist overlaps of many vectors in one call (Sec. III):
numbers of vectors around the batch of one launch (64), the smallest chain,
blocks of every size; against the oracle's direct sum."""
import numpy as np
import pytest

from oracle import basis, twist
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L, K", [(4, 1), (4, 64), (6, 65), (10, 129), (14, 3), (18, 2), (22, 2)])
def test_many_vectors(L, K):
    hs = need_gpu()
    st = basis.enumerate_states(L)
    psi = inputs.gaussian(len(st), 5, K)
    with hs.Chain(L, np.zeros(L), sigma=0.0) as c:
        z = c.twist(to_dev(psi))
    ref = twist.overlap(psi.T, st, L)
    assert (np.abs(z - ref) <= 1e-12 * (psi * psi).sum(1)).all()
