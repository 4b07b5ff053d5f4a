"""GPU parity of the cluster form of MINRES (Algorithm 2 inside one
thread-block cluster, chains of up to 16384 rows): iterates element by element
against the oracle for every cluster size, within the bounds that
test_gpu_minres.py derives for the same recurrence at L = 6..12, or, where the
problem itself amplifies rounding further (Jacobi with a_ii near sigma, alpha_1
near zero at n = 6), no further from the oracle than twice what the grid form
of the same recurrence is."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import hamiltonian, minres
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, torch
from tests.test_gpu_minres import TOL32, TOL64, separated_sigma

pytestmark = pytest.mark.gpu


# (L, CTAs): one thread with rows (n = 6, 20), rows that do not divide by the
# cluster, one to eight rows per thread, CTAs without rows (n = 6 on 8)
@pytest.mark.parametrize("L, cs", [(4, 1), (4, 8), (6, 1), (6, 16), (8, 1), (8, 2), (8, 16), (10, 1),
                                   (10, 4), (12, 1), (12, 2), (12, 4), (12, 8), (12, 16), (14, 4),
                                   (14, 8), (14, 16), (16, 16)])
@pytest.mark.parametrize("kind", ["id", "jacobi", "row"])
def test_iterates_match_oracle(L, cs, kind, monkeypatch):
    hs = need_gpu()
    monkeypatch.setenv("HS_MINRES_CLUSTER", str(cs))
    hv = inputs.disorder(L, 3.0, 0)
    H, diag, st = hamiltonian.build(L, hv)
    n = len(st)
    sigma = separated_sigma(diag)
    A = (H - sigma * sp.identity(n)).tocsr()
    b = inputs.gaussian(n, 11)
    M = hamiltonian.precond_diag(H, diag, sigma, kind)
    def off(k, solve, rhs):
        x, info = solve(rhs, tol=0.0, kmax=k, precond=kind, allow_not_converged=True)
        assert info["iters"] == k and info["form"] == hs.FORM_SMEM
        return np.abs(x.cpu().double().numpy() - xr).max()

    with hs.Chain(L, hv, sigma=sigma) as c:
        for k in (1, 2, 3, 7):
            if k > max(1, n // 4):
                continue
            xr, kr, phir = minres.pminres(A, b, 1.0 / M, kmax=k, tol=0.0)
            scale = np.abs(xr).max()
            for solve, rhs, tol in ((c.minres, to_dev(b), TOL64[k]),
                                    (c.minres_f32, to_dev(b, torch.float32), TOL32[k])):
                if L == 16 and solve == c.minres and kind != "jacobi":
                    continue        # FP64 above 4096 rows: the grid forms
                got = off(k, solve, rhs)
                if got > tol * scale:
                    with monkeypatch.context() as grid:
                        grid.setenv("HS_MINRES_PIPE", "0")
                        assert got <= 2 * off(k, solve, rhs), (L, cs, kind, k, got / scale)


@pytest.mark.parametrize("L, cs", [(4, 1), (8, 1), (10, 2), (12, 8), (14, 16)])
def test_whole_solve_and_edges(L, cs, monkeypatch):
    """A solve to the default tolerance (true residual by the oracle's A), a
    zero and a NaN right-hand side, kmax = 1, and a solve after each of them."""
    hs = need_gpu()
    monkeypatch.setenv("HS_MINRES_CLUSTER", str(cs))
    hv = inputs.disorder(L, 3.0, L)
    H, diag, st = hamiltonian.build(L, hv)
    sigma = 0.1234
    A = (H - sigma * sp.identity(len(st))).tocsr()
    b = inputs.gaussian(len(st), 3)
    M = hamiltonian.precond_diag(H, diag, sigma, "row")
    bad = b.copy()
    bad[len(b) // 2] = np.nan
    with hs.Chain(L, hv, sigma=sigma) as c:
        for _ in range(2):
            x, info = c.minres(to_dev(b), tol=1e-12)
            r = b - A @ x.cpu().numpy()
            assert np.sqrt(r @ (r / M)) <= 5e-12 * np.sqrt(b @ (b / M))
            x, info = c.minres(torch.zeros(len(b), dtype=torch.float64, device="cuda"))
            assert info["iters"] == 0 and not x.abs().max().item()
            with pytest.raises(hs.HSError) as e:
                c.minres(to_dev(bad))
            assert e.value.status == hs.HS_NONFINITE
            x, info = c.minres(to_dev(b), kmax=1, allow_not_converged=True)
            assert info["iters"] == 1
