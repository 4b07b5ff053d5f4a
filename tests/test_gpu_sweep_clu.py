"""hs_sweep on thread-block clusters (chains of up to 4096 rows) and its way back to
the groups of CTAs, against dense eigenvalues of the oracle's H."""
import functools
import json

import numpy as np
import pytest

from oracle import hamiltonian
from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def tune_file(tmp_path, monkeypatch):
    p = tmp_path / "tune.json"
    monkeypatch.setenv("HS_SWEEP_TUNE", str(p))
    return p


@functools.lru_cache(maxsize=None)
def _spectrum(L, seed):
    w = np.linalg.eigvalsh(hamiltonian.build(L, inputs.disorder(L, 3.0, seed))[0].toarray())
    return w[np.lexsort((w, np.abs(w - 0.5 * (w[0] + w[-1]))))]


def _sweep(hs, Ls, K):
    ev, res, z, zz, info = hs.sweep(Ls, [inputs.disorder(L, 3.0, 70 + r) for r, L in enumerate(Ls)], K)
    assert info["converged"] == len(Ls)
    for r, L in enumerate(Ls):
        assert np.abs(ev[r] - _spectrum(L, 70 + r)[:K]).max() < 1e-10
    return info


@pytest.mark.parametrize("refused", ["size", "cache"])
def test_refused_clusters(refused, tune_file, monkeypatch):
    """A cluster size that no launch takes: the groups of CTAs run the sweep; a cached
    size above the largest cluster is timed again."""
    hs = need_gpu()
    Ls = [8, 10, 8, 10]
    if refused == "size":
        monkeypatch.setenv("HS_MINRES_CLUSTER", "32")
    else:
        sm = torch.cuda.get_device_properties(0).multi_processor_count
        tune_file.write_text("{\n" + ",\n".join(
            f'"L{L}_pc2_f64_clu_sm{sm}": {{"S": 64, "one": 0, "rate": 1}}' for L in (8, 10)) + "\n}\n")
    info = _sweep(hs, Ls, 3)
    assert info["tuned"] == [1, 1]
    keys = json.loads(tune_file.read_text())
    assert any("clu" not in k for k in keys) == (refused == "size")
    assert all(v["S"] <= 16 for k, v in keys.items() if "clu" in k)


@pytest.mark.parametrize("cs", [None, "4", "16"])
def test_longest_with_short_chains(cs, tune_file, monkeypatch):
    """Chains of 3432 rows (all compute warps of a CTA at work) and of 70 in one list,
    more of them than clusters at a time run side by side."""
    hs = need_gpu()
    if cs:
        monkeypatch.setenv("HS_MINRES_CLUSTER", cs)
    info = _sweep(hs, [14, 8, 14] + [8] * 40, 3)
    assert cs is None or info["S"] == [int(cs)] * 2


def test_stops_at_the_same_step_as_the_groups(tune_file, monkeypatch):
    """The convergence test on T_k follows every step in both forms: one realisation
    at a time, ten pairs to a loose tolerance (two or more of them often converge in
    one step), the same number of Lanczos steps."""
    hs = need_gpu()
    for r in range(6):
        h = inputs.disorder(10, 3.0, 90 + r)
        with monkeypatch.context() as m:
            m.setenv("HS_SWEEP_S", "8")
            groups = hs.sweep([10], [h], 10, tol=1e-2)[-1]
        clusters = hs.sweep([10], [h], 10, tol=1e-2)[-1]
        assert clusters["max_steps"] == groups["max_steps"]
        assert clusters["converged"] == groups["converged"] == 1
