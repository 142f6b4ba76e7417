"""A run that device memory does not suffice for fails with HAC_ENOMEM and leaves the
handle usable: with memory back, the next run on it goes through, whichever of
the cache's allocations had failed."""
import numpy as np
import pytest

from paper_2106_04727_gb300 import hac

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def test_cache_tables(monkeypatch):
    monkeypatch.setenv("HAC_DENSE_K", "0")
    n = 4_000_000
    X = np.random.RandomState(2).uniform(size=(n, 2)).astype(np.float32)
    hac.cluster(X[:5000], "complete", cache_slots=1)   # the module is loaded
    torch.cuda.empty_cache()
    # tables 92 MiB, queue of insertions 320 MB with a byte per cluster at its end,
    # then the big pairs' buffers
    failed = 0
    ballast = torch.empty(torch.cuda.mem_get_info()[0] - 6000 * MB, dtype=torch.uint8,
                          device="cuda")
    try:
        for left in [40, 80, 120, 200, 340] + list(range(384, 416, 2)) + [500, 700]:
            h = hac.hac_create(X, "complete")
            rest = None
            try:
                rest = torch.empty(torch.cuda.mem_get_info()[0] - left * MB, dtype=torch.uint8,
                                   device="cuda")
                rc = hac.hac_run(h, cache_slots=1, max_rounds=1)
                assert rc in (hac.HAC_ENOMEM, hac.HAC_ETIMEOUT)
                failed += rc == hac.HAC_ENOMEM
                del rest
                rest = None
                torch.cuda.empty_cache()
                assert hac.hac_run(h, cache_slots=1, max_rounds=1) == hac.HAC_ETIMEOUT, left
            finally:
                del rest
                torch.cuda.empty_cache()
                hac.hac_destroy(h)
    finally:
        del ballast
        torch.cuda.empty_cache()
    assert failed > 10
