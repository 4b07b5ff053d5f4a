"""Extremal eigenvalues (hs_extremal) where the short route, one traced Lanczos run per
chain in a cluster, does not end well: the plain recurrence takes over."""
import numpy as np
import pytest

from oracle import hamiltonian
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-3, 1.0, 1e105, 1e120])
def test_extremes_of_large_fields(scale):
    """E_min and E_max of chains whose fields dwarf the exchange: the ends of the
    spectrum by dense eigenvalues, relative to its width."""
    hs = need_gpu()
    L = 8
    hv = inputs.disorder(L, 3.0, 4) * scale
    w = np.linalg.eigvalsh(hamiltonian.build(L, hv)[0].toarray())
    with hs.Chain(L, hv, sigma=0.0) as c:
        emin, emax, mid = c.extremal()
    assert max(abs(emin - w[0]), abs(emax - w[-1]),
               abs(mid - 0.5 * (w[0] + w[-1]))) <= 1e-10 * (w[-1] - w[0])


@pytest.mark.parametrize("L", [8, 12])
def test_extremes_under_a_wait_limit(L, monkeypatch):
    """A wait limit of zero polls stops the traced run; the extremes are still
    right, alone and as the sigma of a chain."""
    hs = need_gpu()
    hv = inputs.disorder(L, 3.0, 4)
    w = np.linalg.eigvalsh(hamiltonian.build(L, hv)[0].toarray())
    monkeypatch.setenv("HS_BARRIER_LIMIT", "0")
    with hs.Chain(L, hv) as c:
        emin, emax, mid = c.extremal()
        assert max(abs(emin - w[0]), abs(emax - w[-1])) <= 1e-10 * (w[-1] - w[0])
        assert abs(c.sigma - 0.5 * (w[0] + w[-1])) <= 1e-10 * (w[-1] - w[0])


@pytest.mark.parametrize("nsm", [1, 3, 0])
def test_extremes_within_an_sm_share(nsm):
    """The extremes with the handle held to a share of the SMs (at L = 14 a cluster
    of one or two CTAs cannot hold the rows, and the plain recurrence runs)."""
    hs = need_gpu()
    for L in (8, 12, 14):
        hv = inputs.disorder(L, 3.0, 4)
        with hs.Chain(L, hv, sigma=0.0) as c:
            ref = c.extremal()
            c.set_sm_budget(nsm)
            got = c.extremal()
        assert max(abs(a - b) for a, b in zip(got, ref)) <= 1e-10 * (ref[1] - ref[0])
