"""CPU check of the six-low-bit superblock H x (sb6.cuh): its plan builder, flat
pass and per-lane row code, run on the CPU by tests/host/sb6_host_check.cu in the
kernel's order with NaN in everything that must not be read, against the
oracle's explicit sparse H of Eq. (1)."""
import os
import subprocess

import numpy as np
import pytest

from oracle import hamiltonian
from paper_2203_09732_gb300 import inputs
from tests.test_sb_host import HERE, _nvcc


@pytest.fixture(scope="module")
def rows_prog(tmp_path_factory):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    out = tmp_path_factory.mktemp("sb6host") / "sb6_host_check"
    src = os.path.join(HERE, "host", "sb6_host_check.cu")
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-O2", "-o", str(out), src],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return str(out)


# (L, KS): KS - 6 mid bits, L - KS top bits: one mid bit, two top bits, the
# library's windows, windows wider than half the chain (classes that are missing)
@pytest.mark.parametrize("L,KS", [(10, 7), (10, 8), (12, 7), (12, 10), (14, 8), (14, 12), (16, 9),
                                  (16, 14), (18, 13), (18, 14), (20, 10), (22, 12), (24, 13),
                                  (24, 14)])
def test_rows_vs_explicit_matrix(rows_prog, tmp_path, L, KS):
    """Every row in FP64 (1e-14 of the row scale, as in test_sb_host.py) and FP32 (the
    rounding bound of an FP32 row sum)."""
    h = np.asarray(inputs.disorder(L, 3.0, 3 * L + KS), dtype=np.float64)
    H, diag, st = hamiltonian.build(L, h)
    x = inputs.gaussian(len(st), 5 + L)
    h.tofile(tmp_path / "h.bin")
    x.tofile(tmp_path / "x.bin")
    sigma = -0.29
    ref = H @ x - sigma * x
    x32 = x.astype(np.float32).astype(np.float64)
    ref32 = H @ x32 - sigma * x32
    bound32 = (L + 4) * 2.0 ** -24 * (np.abs(diag - sigma) * np.abs(x32) + abs(H) @ np.abs(x32)) * 2
    scale = np.abs(diag * x).max() + np.abs(x).max() * L
    r = subprocess.run([rows_prog, str(L), str(KS), repr(sigma), str(tmp_path)],
                       capture_output=True, text=True)
    assert r.returncode == 0, (r.stdout, r.stderr)
    y64 = np.fromfile(tmp_path / "y64.bin")
    y32 = np.fromfile(tmp_path / "y32.bin")
    assert np.isfinite(y64).all() and np.isfinite(y32).all()
    assert np.abs(y64 - ref).max() <= 1e-14 * scale
    assert (np.abs(y32 - ref32) <= bound32 + 1e-30).all()


def test_plan_rejects_splits_out_of_range(rows_prog, tmp_path):
    """No mid bit, more than 8, or fewer than two top bits: no plan."""
    L = 16
    np.asarray(inputs.disorder(L, 1.0, 1), dtype=np.float64).tofile(tmp_path / "h.bin")
    for KS in (6, 15, 16):
        r = subprocess.run([rows_prog, str(L), str(KS), "0.0", str(tmp_path)],
                           capture_output=True, text=True)
        assert r.returncode == 4 and "does not apply" in r.stdout
