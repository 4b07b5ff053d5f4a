"""GPU parity of the row form of MINRES (Algorithm 2 on the whole grid, one to
three rows per thread): iterates element by element against the oracle over one,
two and three rows per thread, CTAs without rows and short last CTAs, within the
bounds that test_gpu_minres.py derives for the same recurrence at L = 6..12, or,
where the problem itself amplifies rounding further, no further from the oracle
than twice what the two-reduction grid form is; the wait limit."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import hamiltonian, minres
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, torch
from tests.test_gpu_minres import TOL32, TOL64, separated_sigma

pytestmark = pytest.mark.gpu


@pytest.fixture
def row(monkeypatch):
    monkeypatch.setenv("HS_MINRES_ROW", "1")
    monkeypatch.setenv("HS_MINRES_CLUSTER", "0")


# (L, SMs): n = 70, 252 and 924 on all SMs (CTAs of few rows, CTAs without rows),
# 12870 rows on 11 (1170 each: three per thread), 16, 31 and all SMs
@pytest.mark.parametrize("L, nsm", [(8, 0), (10, 0), (12, 0), (12, 1), (12, 2), (14, 3), (14, 0),
                                    (16, 11), (16, 16), (16, 31), (16, 0), (18, 0)])
@pytest.mark.parametrize("kind", ["id", "jacobi", "row"])
def test_iterates_match_oracle(L, nsm, kind, row, monkeypatch):
    hs = need_gpu()
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
        c.set_sm_budget(nsm)
        for k in (1, 2, 3, 7):
            xr, kr, phir = minres.pminres(A, b, 1.0 / M, kmax=k, tol=0.0)
            scale = np.abs(xr).max()
            for solve, rhs, tol in ((c.minres, to_dev(b), TOL64[k]),
                                    (c.minres_f32, to_dev(b, torch.float32), TOL32[k])):
                got = off(k, solve, rhs)
                if got > tol * scale:
                    with monkeypatch.context() as grid:
                        grid.setenv("HS_MINRES_ROW", "0")
                        grid.setenv("HS_MINRES_PIPE", "0")
                        c.set_sm_budget(0)
                        assert got <= 2 * off(k, solve, rhs), (L, nsm, kind, k, got / scale)
                        c.set_sm_budget(nsm)


def test_whole_solve_edges_and_wait_limit(row, monkeypatch):
    """A whole solve (true residual by the oracle's A), a NaN right-hand side, a wait
    limit of zero polls (HS_TIMEOUT, no fault), and a solve after each."""
    hs = need_gpu()
    L = 14
    hv = inputs.disorder(L, 3.0, 3)
    H, diag, st = hamiltonian.build(L, hv)
    sigma = 0.1234
    A = (H - sigma * sp.identity(len(st))).tocsr()
    M = hamiltonian.precond_diag(H, diag, sigma, "row")
    b = inputs.gaussian(len(st), 3)
    bad = b.copy()
    bad[5] = np.nan
    with hs.Chain(L, hv, sigma=sigma) as c:
        def solve():
            x, info = c.minres(to_dev(b), tol=1e-12)
            r = b - A @ x.cpu().numpy()
            assert np.sqrt(r @ (r / M)) <= 5e-12 * np.sqrt(b @ (b / M))
        solve()
        x, info = c.minres(torch.zeros(len(b), dtype=torch.float64, device="cuda"))
        assert info["iters"] == 0 and not x.abs().max().item()
        with pytest.raises(hs.HSError) as e:
            c.minres(to_dev(bad))
        assert e.value.status == hs.HS_NONFINITE
        solve()
        with monkeypatch.context() as m:
            m.setenv("HS_BARRIER_LIMIT", "0")
            with pytest.raises(hs.HSError) as e:
                c.minres(to_dev(b))
            assert e.value.status == hs.HS_TIMEOUT
        solve()


def test_default_l18_l20():
    """The default at L = 18 and 20 in both precisions: the reported residual of a
    capped solve falls and the iterates agree with the grid form's."""
    hs = need_gpu()
    for L in (18, 20):
        hv = inputs.disorder(L, 3.0, 1)
        with hs.Chain(L, hv, sigma=0.1234) as c:
            b = to_dev(inputs.gaussian(c.n, 5))
            for f32 in (False, True):
                solve = c.minres_f32 if f32 else c.minres
                rhs = b.float() if f32 else b
                x, info = solve(rhs, tol=0.0, kmax=20, allow_not_converged=True)
                assert info["form"] in (hs.FORM_SMEM, hs.FORM_SMEM1)
                assert info["form"] == hs.FORM_SMEM or (L == 18 and not f32)
                assert info["iters"] == 20 and info["phi"] < 0.9
                with pytest.MonkeyPatch.context() as m:
                    m.setenv("HS_MINRES_ROW", "0")
                    m.setenv("HS_MINRES_PIPE", "0")
                    y, _ = solve(rhs, tol=0.0, kmax=20, allow_not_converged=True)
                d = (x - y).abs().max().item() / y.abs().max().item()
                assert d <= (TOL32 if f32 else TOL64)[20]
