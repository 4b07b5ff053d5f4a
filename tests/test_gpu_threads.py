"""Host threads that use the same kernels with different amounts of shared memory
(chains of different lengths, a handle and a stream each): every call takes the
route, and gives the bits, that it does alone."""
import threading

import numpy as np
import pytest

from paper_2203_09732_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


def _together(jobs, reps):
    """jobs: functions of a stream that return a list of arrays; each alone first, then
    all at once, reps times each. Errors and differences."""
    alone = [job(torch.cuda.Stream()) for job in jobs]
    wrong = []
    start = threading.Barrier(len(jobs))

    def worker(i):
        s = torch.cuda.Stream()
        try:
            start.wait()
            for rep in range(reps):
                for a, b in zip(alone[i], jobs[i](s)):
                    if not np.array_equal(a, b):
                        wrong.append((i, rep, float(np.abs(a - b).max())))
        except Exception as e:
            wrong.append((i, repr(e)))

    th = [threading.Thread(target=worker, args=(i,)) for i in range(len(jobs))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    return wrong


def test_cluster_solves_of_four_lengths():
    hs = need_gpu()

    def solve(L):
        hv, b = inputs.disorder(L, 3.0, L), inputs.gaussian(inputs.dim(L), 3)

        def job(s):
            with torch.cuda.stream(s), hs.Chain(L, hv, sigma=0.1234, stream=s) as c:
                rhs = to_dev(b)
                return [c.minres(rhs, tol=0.0, kmax=12, allow_not_converged=True)[0].cpu().numpy()
                        for _ in range(40)]
        return job

    assert not _together([solve(L) for L in (8, 10, 12, 14)], 4)


def test_twists_of_three_lengths():
    hs = need_gpu()

    def overlap(L):
        hv = inputs.disorder(L, 3.0, L)
        psi = inputs.gaussian(inputs.dim(L), 7)
        psi /= np.linalg.norm(psi)

        def job(s):
            with torch.cuda.stream(s), hs.Chain(L, hv, sigma=0.0, stream=s) as c:
                v = to_dev(psi[None])
                return [np.asarray(c.twist(v)) for _ in range(60)]
        return job

    assert not _together([overlap(L) for L in (20, 22, 24)], 2)


def test_cluster_sweeps_of_different_lengths(tmp_path, monkeypatch):
    hs = need_gpu()
    monkeypatch.setenv("HS_SWEEP_TUNE", str(tmp_path / "tune.json"))

    def sweep(Ls):
        fields = [inputs.disorder(L, 3.0, 30 + r) for r, L in enumerate(Ls)]

        def job(s):
            ev, res, z, zz, info = hs.sweep(Ls, fields, 3)
            assert info["converged"] == len(Ls)
            return [ev, z]
        return job

    assert not _together([sweep([8] * 3), sweep([10, 12]), sweep([14])], 3)
