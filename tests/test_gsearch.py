"""The grouped search (csrc/hac_gsearch.cu) of Ward and avg-2 in runs above the
one-launch capacity, and of complete and average linkage's first round: groups
of 4 and, from 40,000 terminals, of 32 in d <= 2 and 8 above, in every
dimension it takes, ragged group and bucket ends, ties and near ties (left to
the warp-per-terminal FP64 search)."""
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


@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("d", list(range(1, 9)))
def test_every_dimension(lk, d):
    """n = 4,097 + 7 d: groups of 4, most with a ragged last one."""
    dt = np.float32 if d % 2 else np.float64
    X = inputs.gaussian_mixture(4097 + 7 * d, d, 9, seed=50 + d, dtype=dt)
    _check(hac.cluster(X, lk), oracle.rounds(X.astype(np.float64), lk))


@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("name,n", [("gmm5d_1m_f32", 50_003), ("gaussiandisc2d_1m_f32", 70_001),
                                    ("uniformfill5d_1m_f32", 41_000)])
def test_wide_groups(lk, name, n):
    """Groups of 32 (2-D) or 8 (5-D) in the first rounds, of 4 later."""
    X = inputs.workload(name, n=n)
    want = oracle.parchain_cpu(X.astype(np.float64), lk)
    _check(hac.cluster(X, lk), want)


def _one_by_one(X, lk, prec=hac.PREC_F64):
    """The same through an engine, whose searches take one terminal per warp."""
    h = hac.hac_create(X, lk)
    try:
        assert hac.hac_run_batch([h], precision=prec, cache_slots=64) == hac.HAC_OK
        return dict(hac.result_dict(hac.hac_dendrogram(h, len(X))),
                    round=hac.hac_merge_rounds(h, len(X)).astype(np.int64))
    finally:
        hac.hac_destroy(h)


@pytest.mark.parametrize("lk,prec", [("ward", hac.PREC_F64), ("average_sq", hac.PREC_F64),
                                     ("complete", hac.PREC_F64), ("average", hac.PREC_F64),
                                     ("complete", hac.PREC_F32_RECHECK),
                                     ("average", hac.PREC_F32_RECHECK)])
@pytest.mark.parametrize("d", list(range(1, 9)))
def test_wide_groups_in_every_dimension(d, lk, prec):
    """n = 40,001 + 10 d: groups of 32 (d <= 2) or 8 with a ragged last one."""
    dt = np.float64 if d % 2 else np.float32
    X = inputs.gaussian_mixture(40_001 + 10 * d, d, 30, seed=90 + d, dtype=dt)
    got = hac.cluster(X, lk, precision=prec, cache_slots=64)
    closed = lk in LKS   # (the others' FP64 searches take seconds in an engine)
    _check(got, _one_by_one(X, lk, hac.PREC_F64 if closed else hac.PREC_F32_RECHECK),
           rtol=1e-9 if closed else 2e-5)


@pytest.mark.parametrize("lk", ["ward", "average_sq", "complete"])
@pytest.mark.parametrize("kind,d", [("lattice", 2), ("duplicates", 3), ("outliers", 4),
                                    ("clipped", 2), ("gap", 2), ("gap", 5)])
def test_hard_inputs_in_wide_groups(lk, kind, d):
    n = 41_007
    if kind == "lattice":
        X = inputs.lattice(n, d, seed=2, levels=300)
    elif kind == "duplicates":
        X = np.repeat(inputs.gaussian_mixture(n // 3, d, 9, seed=7), 3, axis=0)
        X = np.concatenate([X, X[:n - len(X)]])
    elif kind == "clipped":
        X = inputs.uniform_cube(n, d, seed=21, dtype=np.float32)
        X[:20_000, 1] = 1.0
    elif kind == "gap":
        X = inputs.uniform_cube(n, d, seed=22, dtype=np.float32)
        X[:30_000] = np.float32(0.498) + X[:30_000] * np.float32(0.004)
    else:
        X = np.concatenate([1e-3 * inputs.gaussian_mixture(n - 2, d, 6, seed=3),
                            np.full((1, d), 1e5, np.float32), np.full((1, d), -3e4, np.float32)])
    if lk == "complete":
        _check(hac.cluster(X, lk, precision=hac.PREC_F32_RECHECK, cache_slots=64),
               _one_by_one(X, lk, hac.PREC_F32_RECHECK), rtol=2e-5)
    else:
        _check(hac.cluster(X, lk), _one_by_one(X, lk), rtol=1e-12)


@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("kind", ["lattice", "duplicates", "line", "outliers", "clipped", "gap"])
def test_hard_inputs(lk, kind):
    """The same tree as with every cluster scanned in FP64 (no pruning, no
    grouping)."""
    if kind == "lattice":
        X = inputs.lattice(5000, 2, seed=2, levels=40)
    elif kind == "duplicates":
        X = np.repeat(inputs.gaussian_mixture(450, 3, 5, seed=7), 10, axis=0)
    elif kind == "line":
        X = np.arange(4500, dtype=np.float32)[:, None] * np.float32(0.5)
    elif kind == "clipped":  # points alone in their bucket beside a dense line
        X = inputs.uniform_cube(6000, 2, seed=21, dtype=np.float32)
        X[:3000, 1] = 1.0
    elif kind == "gap":  # groups whose box holds a dense region none of them reaches
        X = inputs.uniform_cube(6000, 2, seed=22, dtype=np.float32)
        X[:4000] = np.float32(0.498) + X[:4000] * np.float32(0.004)
    else:
        X = np.concatenate([1e-3 * inputs.gaussian_mixture(4600, 4, 6, seed=3),
                            np.full((1, 4), 1e5, np.float32), np.full((1, 4), -3e4, np.float32)])
    _check(hac.cluster(X, lk), hac.cluster(X, lk, no_prune=True), rtol=1e-12)


@pytest.mark.parametrize("prec", [hac.PREC_F64, hac.PREC_F32_RECHECK], ids=["f64", "f32recheck"])
@pytest.mark.parametrize("lk", ["complete", "average"])
@pytest.mark.parametrize("d", list(range(1, 9)))
def test_single_points(lk, d, prec, monkeypatch):
    """The first round of complete and average linkage (no dense matrix)."""
    monkeypatch.setenv("HAC_DENSE_K", "0")
    X = inputs.gaussian_mixture(2500 + 7 * d, d, 9, seed=70 + d,
                                dtype=np.float64 if d % 2 else np.float32)
    got = hac.cluster(X, lk, precision=prec, cache_slots=16)
    _check(got, oracle.rounds(X.astype(np.float64), lk),
           rtol=1e-9 if prec == hac.PREC_F64 else 1e-5)


@pytest.mark.parametrize("lk", ["complete", "average"])
def test_single_points_ties(lk, monkeypatch):
    monkeypatch.setenv("HAC_DENSE_K", "0")
    X = inputs.lattice(3000, 2, seed=12, levels=30)
    got = hac.cluster(X, lk, precision=hac.PREC_F32_RECHECK, cache_slots=16)
    _check(got, hac.cluster(X, lk, cache_slots=16), rtol=1e-5)
