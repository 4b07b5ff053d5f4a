"""MINRES of Algorithm 2 on right-hand sides far from 1: the iterates
scale with b, as long as b . M^-1 b is a normal number. Scaling by a power of two
changes no rounding, so the bounds are those of the unscaled iterates against the
oracle (test_gpu_minres.py, test_gpu_minres_pipe.py)."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import hamiltonian, minres
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev
from tests.test_gpu_minres import TOL64, separated_sigma
from tests.test_gpu_minres_pipe import TOL64 as TOL64_ONE

pytestmark = pytest.mark.gpu

FORMS = {"cluster": {}, "row": {"HS_MINRES_CLUSTER": "0", "HS_MINRES_ROW": "1"},
         "one reduction": {"HS_MINRES_PIPE": "1"},
         "grid": {"HS_MINRES_CLUSTER": "0", "HS_MINRES_ROW": "0", "HS_MINRES_PIPE": "0"}}


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("e", [-480, -366, -330, 329, 366, 480])
@pytest.mark.parametrize("kind", ["id", "row"])
def test_scaled_right_hand_side(form, e, kind, monkeypatch):
    hs = need_gpu()
    for k, v in FORMS[form].items():
        monkeypatch.setenv(k, v)
    L = 10
    hv = inputs.disorder(L, 3.0, 0)
    H, diag, st = hamiltonian.build(L, hv)
    sigma = separated_sigma(diag)
    A = (H - sigma * sp.identity(len(st))).tocsr()
    b = inputs.gaussian(len(st), 11)
    M = hamiltonian.precond_diag(H, diag, sigma, kind)
    tol = TOL64_ONE if form == "one reduction" else TOL64
    with hs.Chain(L, hv, sigma=sigma) as c:
        for k in (1, 2, 3, 7):
            xr, _, _ = minres.pminres(A, b, 1.0 / M, kmax=k, tol=0.0)
            x, info = c.minres(to_dev(np.ldexp(b, e)), tol=0.0, kmax=k, precond=kind,
                               allow_not_converged=True)
            assert info["iters"] == k
            got = np.ldexp(x.cpu().numpy(), -e)
            assert np.abs(got - xr).max() <= tol[k] * np.abs(xr).max(), (form, e, kind, k)
