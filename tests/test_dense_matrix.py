"""The position-ordered dense matrix (csrc/hac_dense.cu): complete linkage from
the first round on, the fill from singletons, the compacted rebuild after every
round and the one-launch rounds at its end, for both linkages, against the CPU
oracle merge for merge and round for round."""
import numpy as np
import pytest

import oracle
from paper_2106_04727_gb300 import hac, inputs

pytestmark = pytest.mark.gpu

PRECS = [hac.PREC_F64, hac.PREC_F32_RECHECK]
PREC_IDS = ["f64", "f32recheck"]


def _check(got, want, rtol):
    c = oracle.compare(got, want, rtol=rtol)
    assert c["ok"], c
    key = lambda t: sorted(zip(t["round"].tolist(), t["a"].tolist(), t["b"].tolist()))
    assert key(got) == key(want)


# 32-wide tiles, 64-entry row steps, the row stride's padding to 4, block counts
# (64, 200 clusters) and the one-launch capacity (1,024)
@pytest.mark.parametrize("prec", PRECS, ids=PREC_IDS)
@pytest.mark.parametrize("n,d,dt", [
    (2, 1, np.float32), (3, 2, np.float64), (31, 3, np.float32), (33, 5, np.float64),
    (64, 16, np.float32), (65, 8, np.float64), (201, 4, np.float32), (257, 10, np.float64),
    (1024, 2, np.float64), (1027, 7, np.float32), (2500, 3, np.float64), (4001, 12, np.float32)])
def test_complete_from_first_round(n, d, dt, prec):
    X = inputs.gaussian_mixture(n, d, 5, seed=n * 13 + d, dtype=dt)
    got = hac.cluster(X, "complete", precision=prec, cache_slots=64)
    _check(got, oracle.rounds(X.astype(np.float64), "complete"),
           1e-9 if prec == hac.PREC_F64 else 1e-5)
    st = got["stats"]
    assert st["dense_k"] == n and st["dense_rounds"] == st["rounds"]
    assert st["dense_point_pairs"] == n * (n - 1) // 2


@pytest.mark.parametrize("prec", PRECS, ids=PREC_IDS)
def test_complete_ties(prec):
    """Lattice points: equal distances are decided in FP64 by cid; the FP32 mode
    re-scores and gives exactly the FP64 tree."""
    X = inputs.lattice(600, 3, seed=4, levels=10)
    got = hac.cluster(X, "complete", precision=prec)
    _check(got, oracle.rounds(X.astype(np.float64), "complete"),
           0.0 if prec == hac.PREC_F64 else 1e-5)
    if prec == hac.PREC_F32_RECHECK:
        assert got["stats"]["dense_rechecks"] > 0


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("lk", ["complete", "average"])
def test_many_duplicates(lk, dt):
    """Groups of equal points: their zero distances are exact from the fill, so
    no group is re-scored pair by pair."""
    X = np.repeat(inputs.gaussian_mixture(15, 4, 3, seed=9, dtype=dt), 40, axis=0)
    got = hac.cluster(X, lk, precision=hac.PREC_F32_RECHECK)
    want = hac.cluster(X, lk, precision=hac.PREC_F64)
    _check(got, want, 1e-5)
    assert (got["h"] == 0.0).sum() == 15 * 39
    assert got["stats"]["dense_rechecks"] < 600


@pytest.mark.parametrize("scale", [1e-24, 1e-9, 1e9])
@pytest.mark.parametrize("lk", ["complete", "average"])
def test_scales(lk, scale):
    X = (inputs.gaussian_mixture(500, 3, 4, seed=6, dtype=np.float64) * scale).astype(np.float32)
    want = oracle.rounds(X.astype(np.float64), lk)
    _check(hac.cluster(X, lk, precision=hac.PREC_F64), want, 1e-9)
    _check(hac.cluster(X, lk, precision=hac.PREC_F32_RECHECK), want, 1e-5)


@pytest.mark.parametrize("lk", ["complete", "average"])
def test_round_limits(lk):
    """A limit may stop the one-launch rounds anywhere; a rerun is complete."""
    X = inputs.gaussian_mixture(1500, 2, 4, seed=3)
    want = oracle.rounds(X.astype(np.float64), lk)
    last = int(want["round"].max()) + 1
    h = hac.hac_create(X, lk)
    try:
        for r in (1, last // 2, last - 1):
            assert hac.hac_run(h, max_rounds=r) == hac.HAC_ETIMEOUT
        for kw in (dict(max_rounds=last), dict(timeout_s=60.0), dict(precision=hac.PREC_F32_RECHECK)):
            assert hac.hac_run(h, **kw) == hac.HAC_OK
            m = hac.hac_dendrogram(h, len(X))
            got = dict(a=m["cid_a"], b=m["cid_b"], h=m["height"], size=m["size"],
                       round=hac.hac_merge_rounds(h, len(X)).astype(np.int64))
            _check(got, want, 1e-5 if "precision" in kw else 1e-9)
    finally:
        hac.hac_destroy(h)


def test_more_estimates_in_the_windows_than_a_counter_holds(monkeypatch):
    """46,400 points whose FP32 distances all lie within the error term (set by one
    point far away): 2.15 * 10^9 estimates are listed for an FP64 re-score, pass by
    pass through a list of 4 * 10^6."""
    n, d = 46_400, 16
    monkeypatch.setenv("HAC_DENSE_K", str(n))
    r = np.random.RandomState(11)
    X = r.randint(0, 2, (n, d)) * 2.0**-25 + 2.0**-30 * r.uniform(size=(n, d))
    X[0] = -1.0
    h = hac.hac_create(X, "complete")
    try:  # the first round lists them all
        assert hac.hac_run(h, precision=hac.PREC_F32_RECHECK, max_rounds=1) == hac.HAC_ETIMEOUT
    finally:
        hac.hac_destroy(h)


def test_complete_estimates_are_correctly_rounded():
    """Differences of points of [1, 2) on a line are FP32 numbers, and the rounded root
    of their rounded square is they: every height that was not re-scored is the FP64
    value plus the same bound."""
    X = (1.0 + np.random.RandomState(4).uniform(size=(900, 1))).astype(np.float32)
    got = hac.cluster(X, "complete", precision=hac.PREC_F32_RECHECK)
    want = oracle.nnchain(X.astype(np.float64), "complete")
    assert oracle.compare(got, want, rtol=1e-5)["ok"]
    true = dict(zip(zip(want["a"].tolist(), want["b"].tolist()), want["h"]))
    step = np.array([np.float64(h).view(np.int64) - np.float64(true[a, b]).view(np.int64)
                     for a, b, h in zip(got["a"].tolist(), got["b"].tolist(), got["h"])])
    assert np.count_nonzero(step) > 300
    assert len(np.unique(step[step != 0])) == 1   # the bound is a step of the bit pattern
