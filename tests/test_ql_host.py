"""CPU check of the plane rotation of the sweep's QL iteration (ql.cuh) over the whole
range of doubles, against math.hypot and true quotients."""
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from tests.test_sb_host import HERE, _nvcc

U = 2.0 ** -53


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    out = tmp_path_factory.mktemp("ql") / "ql_host_check"
    src = os.path.join(HERE, "host", "ql_host_check.cu")
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-o", str(out), src], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return str(out)


def _run(prog, pairs):
    r = subprocess.run([prog], input="".join(f"{f.hex()} {g.hex()}\n" for f, g in pairs),
                       capture_output=True, text=True)
    assert r.returncode == 0
    return [tuple(float.fromhex(x) for x in line.split()) for line in r.stdout.splitlines()]


def test_rotation_over_all_exponents(prog):
    """r within 4 units of rounding of the root (a sum of two squares, a root, a product:
    at most 3), s and c within 5 of the true quotients, or the smallest double."""
    rng = np.random.default_rng(1)
    pairs = []
    for e in list(range(-1060, 1020, 10)) + [-541, -540, -539, -482, -481, -480, -479, 499, 500, 501, 511, 512]:
        for d in (0, 0, 1, 7, 30, 60):
            f, g = (float(math.ldexp(rng.uniform(1, 2) * rng.choice([-1, 1]), e - k)) for k in (0, d))
            pairs += [(f, g), (g, f)]
    tiny = 5e-324
    got = _run(prog, pairs)
    assert len(got) == len(pairs)
    for (f, g), (r, s, c) in zip(pairs, got):
        assert abs(r - math.hypot(f, g)) <= 4 * U * r + tiny
        scale = Fraction(math.hypot(f, g))
        for q, x in ((s, f), (c, g)):
            true = Fraction(x) / scale
            assert abs(Fraction(q) - true) <= abs(true) * Fraction(5 * U) + Fraction(tiny)


def test_rotation_of_zeros(prog):
    got = _run(prog, [(0.0, 0.0), (0.0, 3.0), (-2.0, 0.0), (0.0, 1e-200), (1e300, 0.0)])
    assert got == [(0.0, 0.0, 0.0), (3.0, 0.0, 1.0), (2.0, -1.0, 0.0), (1e-200, 0.0, 1.0), (1e300, 1.0, 0.0)]
