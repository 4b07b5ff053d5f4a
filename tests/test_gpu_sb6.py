"""GPU parity of the six-low-bit superblock product (FP64 MINRES pass A from
L = 22 on) on small chains over windows that reach every bond kind, at L = 22 and
24 in full, and of MINRES on it (its default at L = 22)."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import hamiltonian, minres
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, torch
from tests.test_gpu_minres import TOL64, separated_sigma

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L, KS", [(12, 7), (12, 10), (14, 8), (16, 14), (18, 13), (22, 13), (24, 13)])
@pytest.mark.parametrize("shifted", [0, 1])
def test_matvec_vs_explicit_matrix(L, KS, shifted, monkeypatch):
    """Every row within 1e-14 of the row scale (as test_gpu_matvec.py), for vectors
    on and off a 16-byte boundary (equal element for element)."""
    hs = need_gpu()
    monkeypatch.setenv("HS_SB_PLANS", "1")
    monkeypatch.setenv("HS_SB6_KS", str(KS))
    monkeypatch.setenv("HS_HV_SB", "1")
    h = inputs.disorder(L, 3.0, 100 + L)
    H, diag, st = hamiltonian.build(L, h)
    n, sigma = len(st), 0.37
    x = inputs.gaussian(n, 7)
    ref = H @ x - (sigma * x if shifted else 0)
    with hs.Chain(L, h, sigma=sigma) as c:
        y = c.matvec(to_dev(x), shifted=bool(shifted)).cpu().numpy()
        off = to_dev(np.concatenate([[np.nan], x]))[1:]
        z = c.matvec(off, shifted=bool(shifted)).cpu().numpy()
    scale = np.abs(diag * x).max() + np.abs(x).max() * L
    assert np.abs(y - ref).max() <= 1e-14 * scale
    assert np.array_equal(y, z)


@pytest.mark.parametrize("kind", ["id", "row"])
def test_minres_iterates_l22(kind):
    hs = need_gpu()
    L = 22
    hv = inputs.disorder(L, 3.0, 0)
    H, diag, st = hamiltonian.build(L, hv)
    sigma = separated_sigma(diag)
    A = (H - sigma * sp.identity(len(st))).tocsr()
    b = inputs.gaussian(len(st), 11)
    M = hamiltonian.precond_diag(H, diag, sigma, kind)
    with hs.Chain(L, hv, sigma=sigma) as c:
        for k in (1, 3, 7):
            xr, kr, phir = minres.pminres(A, b, 1.0 / M, kmax=k, tol=0.0)
            x, info = c.minres(to_dev(b), tol=0.0, kmax=k, precond=kind, allow_not_converged=True)
            assert info["iters"] == k and info["form"] == hs.FORM_SUPERBLOCK
            assert np.abs(x.cpu().numpy() - xr).max() <= TOL64[k] * np.abs(xr).max()


def test_routes_at_l22():
    """FP64 at L = 22: the two-pass form with the row norm; Jacobi keeps the
    persistent form, also where a_ii - sigma is at the rounding level, which the
    two-pass form refuses."""
    hs = need_gpu()
    L = 22
    hv = inputs.disorder(L, 3.0, 0)
    with hs.Chain(L, hv, sigma=0.0) as c:
        c.sigma = float(c.diag()[0][12345].item()) + 1e-14
        b = to_dev(inputs.gaussian(c.n, 3))
        for kind, form in (("row", hs.FORM_SUPERBLOCK), ("jacobi", hs.FORM_PERSISTENT)):
            x, info = c.minres(b, tol=0.0, kmax=3, precond=kind, allow_not_converged=True)
            assert info["form"] == form and info["iters"] == 3 and torch.isfinite(x).all()
