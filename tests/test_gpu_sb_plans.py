"""Superblock plans made at first use: forms that the environment selects after a
handle was made give the products and iterates of a handle made under that
environment; a first use under stream capture takes the default form."""
import pytest

from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, torch

pytestmark = pytest.mark.gpu

L = 22


def _vectors(n, dtype):
    g = torch.Generator(device="cuda").manual_seed(5)
    return torch.randn(n, generator=g, device="cuda", dtype=dtype)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("form", ["0", "1"])
def test_plans_made_later(dtype, form, monkeypatch):
    hs = need_gpu()
    dt = torch.float32 if dtype == "f32" else torch.float64
    hv = inputs.disorder(L, 3.0, 1)
    got = []
    for when in ("before", "after"):
        with monkeypatch.context() as m:
            env = {"HS_HV_SB": "1", "HS_SB4": form, "HS_MINRES_SB": "1"}
            if when == "before":
                for k, v in env.items():
                    m.setenv(k, v)
            with hs.Chain(L, hv, sigma=0.1) as c:
                x = _vectors(c.n, dt)
                for k, v in env.items():
                    m.setenv(k, v)
                y = c.matvec(x, shifted=True)
                solve = c.minres_f32 if dtype == "f32" else c.minres
                z, info = solve(x, tol=0.0, kmax=5, allow_not_converged=True)
                assert info["form"] == hs.FORM_SUPERBLOCK
                got.append((y.clone(), z.clone()))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])


def test_small_share_takes_the_ten_bit_pass():
    """FP32 solves on fewer than six SMs (L = 24) need the ten-bit plan: made then; the
    iterate is the class form's up to the order of FP32 sums (the bound of
    test_gpu_minres.py at 7 iterations)."""
    hs = need_gpu()
    with hs.Chain(24, inputs.disorder(24, 3.0, 1), sigma=0.1) as c:
        b = _vectors(c.n, torch.float32)
        x = [c.minres_f32(b, tol=0.0, kmax=7, allow_not_converged=True)[0].clone()]
        c.set_sm_budget(5)
        y, info = c.minres_f32(b, tol=0.0, kmax=7, allow_not_converged=True)
        assert info["form"] == hs.FORM_SUPERBLOCK
        assert (x[0] - y).abs().max().item() <= 1e-5 * x[0].abs().max().item()


def test_first_use_under_capture(monkeypatch):
    hs = need_gpu()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s), hs.Chain(L, inputs.disorder(L, 3.0, 1), sigma=0.1, stream=s) as c:
        x = _vectors(c.n, torch.float32)
        y, ref = torch.empty_like(x), torch.empty_like(x)
        c.matvec(x, ref, shifted=True)
        s.synchronize()
        monkeypatch.setenv("HS_HV_SB", "1")
        monkeypatch.setenv("HS_SB4", "1")
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            c.matvec(x, y, shifted=True)
        g.replay()
        s.synchronize()
        assert torch.equal(y, ref)
