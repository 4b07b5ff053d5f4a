"""GPU parity of the one-reduction recurrence on the row layout: iterates element
by element against the oracle over one, two and three rows per thread, CTAs
without rows and short last CTAs, without and with replacement steps (every step,
every fifth), within the bounds that test_gpu_minres_pipe.py derives for the same
recurrence at L = 6..12, or, where the problem itself amplifies rounding further,
no further from the oracle than twice what the two-reduction grid form is; whole
solves, non-finite input and the wait limit."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import hamiltonian, minres
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, torch
from tests.test_gpu_minres import separated_sigma
from tests.test_gpu_minres_pipe import TOL32, TOL64, pipe  # noqa: F401

pytestmark = pytest.mark.gpu


# (L, SMs): 1056 rows at most per CTA; 12870 rows on 13 SMs (990 each: three per
# thread), 19 (678: two), 36 (358: two) and 37 (348: one); on 12 SMs (1073) the
# shared-memory form takes the solve
@pytest.mark.parametrize("L, nsm", [(10, 0), (12, 1), (14, 4), (14, 0), (16, 12), (16, 13),
                                    (16, 19), (16, 36), (16, 37), (16, 0), (18, 0)])
@pytest.mark.parametrize("kind", ["id", "row"])
@pytest.mark.parametrize("R", [0, 1, 5])
def test_iterates_match_oracle(L, nsm, kind, R, pipe, monkeypatch):  # noqa: F811
    hs = need_gpu()
    pipe(R)
    hv = inputs.disorder(L, 3.0, 0)
    H, diag, st = hamiltonian.build(L, hv)
    n = len(st)
    sigma = separated_sigma(diag)
    A = (H - sigma * sp.identity(n)).tocsr()
    b = inputs.gaussian(n, 11)
    M = hamiltonian.precond_diag(H, diag, sigma, kind)

    def off(k, solve, rhs, form):
        x, info = solve(rhs, tol=0.0, kmax=k, precond=kind, allow_not_converged=True)
        assert info["iters"] == k and info["form"] == form
        return np.abs(x.cpu().double().numpy() - xr).max()

    with hs.Chain(L, hv, sigma=sigma) as c:
        c.set_sm_budget(nsm)
        for k in (1, 2, 3, 7):
            xr, kr, phir = minres.pminres(A, b, 1.0 / M, kmax=k, tol=0.0)
            scale = np.abs(xr).max()
            for solve, rhs, tol in ((c.minres, to_dev(b), TOL64[k]),
                                    (c.minres_f32, to_dev(b, torch.float32), TOL32[k])):
                got = off(k, solve, rhs, hs.FORM_SMEM1)
                if got > tol * scale:
                    with monkeypatch.context() as grid:
                        grid.setenv("HS_MINRES_CLUSTER", "0")
                        grid.setenv("HS_MINRES_ROW", "0")
                        grid.setenv("HS_MINRES_PIPE", "0")
                        c.set_sm_budget(0)
                        assert got <= 2 * off(k, solve, rhs, hs.FORM_SMEM), (L, nsm, kind, k)
                        c.set_sm_budget(nsm)


@pytest.mark.parametrize("L, nsm", [(14, 4), (16, 0), (16, 25)])
def test_whole_solve_edges_and_wait_limit(L, nsm, pipe, monkeypatch):  # noqa: F811
    """A whole solve (true residual by the oracle's A, at most 5x the tolerance as
    for the two-reduction form), zero and NaN right-hand sides, a wait limit of
    zero polls (HS_TIMEOUT, no fault), and a solve after each."""
    hs = need_gpu()
    hv = inputs.disorder(L, 3.0, 3)
    H, diag, st = hamiltonian.build(L, hv)
    sigma = 0.1234
    A = (H - sigma * sp.identity(len(st))).tocsr()
    M = hamiltonian.precond_diag(H, diag, sigma, "row")
    b = inputs.gaussian(len(st), 3)
    bad = b.copy()
    bad[len(b) - 1] = np.nan
    with hs.Chain(L, hv, sigma=sigma) as c:
        c.set_sm_budget(nsm)

        def solve():
            x, info = c.minres(to_dev(b), tol=1e-10)
            assert info["form"] == hs.FORM_SMEM1
            r = b - A @ x.cpu().numpy()
            assert np.sqrt(r @ (r / M)) <= 5e-10 * np.sqrt(b @ (b / M))
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
