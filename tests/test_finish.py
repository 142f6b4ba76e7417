"""The one-launch rounds of Ward and avg-2 (csrc/hac_finish.cu): whole runs from
the points, and the last rounds of larger runs, against the CPU oracle merge
for merge and round for round; block counts, the capacity and what lies just
beyond it; ties; scales the FP32 screening would not hold; round limits."""
import numpy as np
import pytest

import oracle
from paper_2106_04727_gb300 import hac, inputs

pytestmark = pytest.mark.gpu

LKS = ["ward", "average_sq"]


def _check(got, want, rtol=1e-9):
    c = oracle.compare(got, want, rtol=rtol)
    assert c["ok"], c
    key = lambda t: sorted(zip(t["round"].tolist(), t["a"].tolist(), t["b"].tolist()))
    assert key(got) == key(want)


# block counts change at 96, 320 and 640 clusters; a block's lists hold 1,024
# threads x 4 entries; d = 16 records allow 2,688 clusters; 4,097 and 2,689
# start with ordinary rounds
@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("n,d,dt", [
    (2, 1, np.float64), (3, 16, np.float32), (32, 2, np.float32), (33, 3, np.float64),
    (96, 5, np.float32), (97, 7, np.float32), (320, 9, np.float64), (321, 11, np.float32),
    (640, 13, np.float32), (641, 4, np.float64), (1025, 6, np.float32), (2688, 16, np.float32),
    (2689, 16, np.float64), (4096, 2, np.float32), (4097, 3, np.float64)])
def test_sizes(lk, n, d, dt):
    X = inputs.gaussian_mixture(n, d, 6, seed=n + d, dtype=dt)
    want = oracle.rounds(X.astype(np.float64), lk)
    for prec in (hac.PREC_F64, hac.PREC_F32_RECHECK):
        _check(hac.cluster(X, lk, precision=prec), want)


@pytest.mark.parametrize("lk", LKS)
def test_ties_and_duplicates(lk):
    """Lattice points with many equal distances (the FP64 pass decides, ties by
    cid): a valid greedy tree, the same in both modes."""
    X = inputs.lattice(700, 2, seed=5, levels=9)
    got = hac.cluster(X, lk)
    bad, stats = oracle.validate(X.astype(np.float64), lk, got, rtol=1e-9, htol=1e-9)
    assert bad == 0, stats
    _check(hac.cluster(X, lk, precision=hac.PREC_F32_RECHECK), got, rtol=0.0)


@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("scale", [1e-11, 1e-8, 1e11, 1e14])
def test_scales(lk, scale):
    """Far from 1 the FP32 squares would flush or overflow: those inputs are
    clustered at another scale; next to the limits the screening still holds."""
    X = inputs.gaussian_mixture(300, 3, 4, seed=8, dtype=np.float64) * (scale / 50.0)
    _check(hac.cluster(X, lk), oracle.rounds(X, lk))


@pytest.mark.parametrize("lk", LKS)
def test_limits_and_bad_input(lk):
    X = inputs.gaussian_mixture(1500, 2, 4, seed=3)
    want = oracle.rounds(X.astype(np.float64), lk)
    last = int(want["round"].max()) + 1
    h = hac.hac_create(X, lk)
    try:
        assert hac.hac_run(h, max_rounds=last - 1) == hac.HAC_ETIMEOUT
        for kw in (dict(max_rounds=last), dict(timeout_s=60.0), {}):
            assert hac.hac_run(h, **kw) == hac.HAC_OK
            m = hac.hac_dendrogram(h, len(X))
            got = dict(a=m["cid_a"], b=m["cid_b"], h=m["height"], size=m["size"],
                       round=hac.hac_merge_rounds(h, len(X)).astype(np.int64))
            _check(got, want)
            st = hac.hac_stats(h)
            assert st["rounds"] == last and st["merges"] == len(X) - 1
    finally:
        hac.hac_destroy(h)
    import torch
    x = torch.full((100, 2), float("nan"), device="cuda")
    h = hac.hac_create_device(x.data_ptr(), 100, 2, np.float32, lk)
    try:
        assert hac.hac_run(h) == hac.HAC_EINVAL
    finally:
        hac.hac_destroy(h)


@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("n,d,one", [(4096, 8, True), (3936, 9, True), (3936, 10, True),
                                     (3937, 10, False), (3392, 11, True), (3392, 12, True),
                                     (3393, 12, False), (2688, 13, True), (2689, 13, False)])
def test_capacities(lk, n, d, one):
    """The most points of a run that is one launch, by dimension, and one more; the
    allocation-free entry point on both sides too."""
    torch = pytest.importorskip("torch")
    X = inputs.gaussian_mixture(n, d, 6, seed=n + d)
    want = oracle.rounds(X.astype(np.float64), lk)
    got = hac.cluster(X, lk, precision=hac.PREC_F32_RECHECK)
    _check(got, want)
    assert (got["stats"]["kernel_launches"] == 1) == one
    src = torch.from_numpy(X).cuda()
    out = torch.zeros((n - 1) * 4, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    for prec in (hac.PREC_F64, hac.PREC_F32_RECHECK):
        assert hac.hac_run_static(src.data_ptr(), n, d, X.dtype, lk, out.data_ptr(), n - 1,
                                  precision=prec) == hac.HAC_OK
        c = oracle.compare(hac.result_dict(out.cpu().numpy().view(hac.MERGE_DTYPE)), want, rtol=1e-9)
        assert c["ok"], c
