"""GPU parity of the class form (FP32 products and MINRES pass A, one warp per block
of ten low bits, CTAs by class): every row of a product within the rounding of its
own sum ((L + 4) u times the sum of its terms' magnitudes) of the oracle's matrix,
from chains where most classes are empty to many blocks per warp; MINRES iterates
within the bounds that test_gpu_minres.py derives for Algorithm 2; small SM
budgets, where pass A goes back to the ten-low-bit superblock form."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import hamiltonian, minres
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, torch
from tests.test_gpu_minres import TOL32, separated_sigma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [12, 14, 16, 18, 20])
@pytest.mark.parametrize("shifted", [False, True])
def test_product_matches_oracle(L, shifted, monkeypatch):
    hs = need_gpu()
    monkeypatch.setenv("HS_KLO", "10")
    monkeypatch.setenv("HS_HV_CLS", "1")
    hv = inputs.disorder(L, 3.0, 7)
    H, diag, st = hamiltonian.build(L, hv)
    n = len(st)
    A = (H - (0.37 if shifted else 0.0) * sp.identity(n)).tocsr()
    xs = [inputs.gaussian(n, 3), np.zeros(n), np.zeros(n)]
    xs[1][n // 3] = 1.0
    with hs.Chain(L, hv, sigma=0.37) as c:
        for x in xs:
            xd = to_dev(x, torch.float32)
            xr = xd.cpu().double().numpy()
            y = torch.full_like(xd, float("nan"))
            c.matvec(xd, y, shifted=shifted)
            # |a_ii - sigma| carries the rounding of its terms: L / 4 + sum |h| / 2 + |sigma|
            mag = abs(A) @ np.abs(xr) + (0.25 * L + 0.5 * np.abs(hv).sum() + 0.37) * np.abs(xr)
            err = np.abs(y.cpu().double().numpy() - A @ xr)
            assert (err <= (L + 4) * 2.0 ** -24 * mag).all(), (L, err.max())


@pytest.mark.parametrize("L", [24, 26])
def test_product_matches_fp64(L):
    """The default at L = 24 and 26 against the FP64 product, row by row."""
    hs = need_gpu()
    hv = inputs.disorder(L, 3.0, 2)
    with hs.Chain(L, hv, sigma=0.37) as c:
        x = torch.randn(c.n, generator=torch.Generator().manual_seed(1)).cuda()
        y = c.matvec(x, shifted=True)
        z = c.matvec(x.double(), shifted=True)
        # off-diagonal magnitudes: (H - sigma) |x| less its diagonal part
        ax = x.double().abs()
        off = c.matvec(ax, shifted=True) - (c.diag()[0] - 0.37) * ax
        mag = off + (0.25 * L + 0.5 * np.abs(hv).sum() + 0.37) * 2 * ax
        assert ((y.double() - z).abs() <= (L + 4) * 2.0 ** -24 * mag).all()


@pytest.mark.parametrize("nsm", [0, 2, 7])
@pytest.mark.parametrize("kind", ["id", "row"])
def test_minres_iterates_match_oracle_l22(nsm, kind, monkeypatch):
    hs = need_gpu()
    monkeypatch.setenv("HS_MINRES_SB", "1")
    L = 22
    hv = inputs.disorder(L, 3.0, 0)
    H, diag, st = hamiltonian.build(L, hv)
    sigma = separated_sigma(diag)
    A = (H - sigma * sp.identity(len(st))).tocsr()
    b = inputs.gaussian(len(st), 11)
    M = hamiltonian.precond_diag(H, diag, sigma, kind)
    with hs.Chain(L, hv, sigma=sigma) as c:
        c.set_sm_budget(nsm)
        for k in (1, 3, 7):
            xr, kr, phir = minres.pminres(A, b, 1.0 / M, kmax=k, tol=0.0)
            x, info = c.minres_f32(to_dev(b, torch.float32), tol=0.0, kmax=k, precond=kind,
                                   allow_not_converged=True)
            assert info["form"] == hs.FORM_SUPERBLOCK and info["iters"] == k
            err = np.abs(x.cpu().double().numpy() - xr).max()
            assert err <= TOL32[k] * np.abs(xr).max(), (kind, k, err / np.abs(xr).max())
