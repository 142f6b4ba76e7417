"""Distinct handles in several host threads at once: every run succeeds and gives
what it gives alone (the launches' shared memory, above 48 KB, is an attribute of
the kernel that all threads share)."""
import threading

import numpy as np
import pytest

from paper_2106_04727_gb300 import hac, inputs

pytestmark = pytest.mark.gpu


def _together(jobs, times):
    """Every job `times` times in its own thread; the exceptions."""
    failed, gate = [], threading.Barrier(len(jobs))

    def loop(job):
        gate.wait()
        for _ in range(times):
            try:
                job()
            except Exception as e:   # noqa: BLE001 (reported by the caller)
                failed.append(repr(e))
                return

    thr = [threading.Thread(target=loop, args=(j,)) for j in jobs]
    for t in thr:
        t.start()
    for t in thr:
        t.join()
    return failed


def _job(X, lk, **kw):
    want = hac.cluster(X, lk, **kw)

    def run():
        got = hac.cluster(X, lk, **kw)
        for f in ("a", "b", "size"):
            assert np.array_equal(got[f], want[f])

    return run


@pytest.mark.parametrize("lk", ["ward", "average_sq"])
def test_one_launch_runs(lk):
    """Staged records of 1,600 to 4,000 clusters: 51 to 128 KB."""
    jobs = [_job(inputs.gaussian_mixture(n, 5, 6, seed=n), lk) for n in (1600, 4000, 2300, 3100)]
    assert _together(jobs, 150) == []


def test_cache_updates(monkeypatch):
    """256 slots a cluster take more than the default 48 KB, 8 and 64 do not."""
    monkeypatch.setenv("HAC_DENSE_K", "0")
    X = inputs.gaussian_mixture(1500, 2, 5, seed=3)
    # (heights, and with them ties, depend on what the cache kept: sizes only)
    jobs = []
    for slots in (256, 8, 256, 64):
        def run(slots=slots):
            got = hac.cluster(X, "complete", cache_slots=slots)
            assert got["size"][-1] == len(X)
        jobs.append(run)
    assert _together(jobs, 60) == []
