"""GPU parity of the one-thread-per-row product: every row within the rounding of
its own sum (at most L + 3 products and additions, so (L + 4) u times the sum of
their magnitudes) of the oracle's matrix, over chains of one block to many, low
parts of 2 to 10 bits, both precisions, with and without the shift."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import hamiltonian
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L, klo", [(4, 0), (6, 0), (8, 0), (10, 0), (12, 0), (12, 2), (12, 10), (14, 0),
                                    (14, 3), (16, 6), (18, 0), (18, 10), (20, 0)])
@pytest.mark.parametrize("shifted", [False, True])
def test_rows_match_oracle(L, klo, shifted, monkeypatch):
    hs = need_gpu()
    if klo:
        monkeypatch.setenv("HS_KLO", str(klo))
    hv = inputs.disorder(L, 3.0, 7)
    H, diag, st = hamiltonian.build(L, hv)
    n = len(st)
    A = (H - (0.37 if shifted else 0.0) * sp.identity(n)).tocsr()
    xs = [inputs.gaussian(n, 3), np.zeros(n), np.zeros(n)]
    xs[1][n // 3] = 1.0
    with hs.Chain(L, hv, sigma=0.37) as c:
        for x in xs:
            for dt, u in ((torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)):
                xd = to_dev(x, dt)
                xr = xd.cpu().double().numpy()
                y = torch.full_like(xd, float("nan"))
                c.matvec(xd, y, shifted=shifted)
                # |a_ii - sigma| carries the rounding of its terms: L / 4 + sum |h| / 2 + |sigma|
                mag = abs(A) @ np.abs(xr) + (0.25 * L + 0.5 * np.abs(hv).sum() + 0.37) * np.abs(xr)
                err = np.abs(y.cpu().double().numpy() - A @ xr)
                assert (err <= (L + 4) * u * mag).all(), (L, klo, dt, err.max())
