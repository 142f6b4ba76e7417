"""The tensor-core screening of the exhaustive search (csrc/hac_brute.cu; Ward
and avg-2 in d > 8, FP32 mode, above the one-launch capacity): the FP64 tree,
whatever the data do to the FP16 products."""
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


# ragged row blocks (256) and tiles (128), every padded dimension class, d <= 8
# through HAC_BRUTE; FP64 input (rounded FP32 copy)
@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("n,d,dt", [(4097, 9, np.float32), (5000, 16, np.float32),
                                    (4353, 12, np.float64), (6001, 10, np.float32),
                                    (4225, 5, np.float32), (4500, 8, np.float64)])
def test_matches_oracle(lk, n, d, dt, monkeypatch):
    monkeypatch.setenv("HAC_BRUTE", "1")
    X = inputs.gaussian_mixture(n, d, 9, seed=n + d, dtype=dt)
    got = hac.cluster(X, lk, precision=hac.PREC_F32_RECHECK)
    _check(got, oracle.rounds(X.astype(np.float64), lk))
    assert got["stats"]["nodes_visited"] == 0
    assert got["stats"]["leaf_tests"] >= got["stats"]["naive_pairs"]


def _hard(kind):
    if kind == "lattice":       # exact ties among singletons
        return inputs.lattice(5000, 16, seed=3, levels=16)
    if kind == "tight":         # clusters far tighter than FP16 resolves from the centre
        X = inputs.gaussian_mixture(4800, 12, 8, seed=5, sigma_lo=1e-3, sigma_hi=2e-3)
        return np.concatenate([X, np.full((1, 12), 3e4, np.float32)])
    if kind == "one_spot":      # everything in one spot but a few outliers
        X = 100.0 + 1e-2 * inputs.gaussian_mixture(4700, 10, 1, seed=6).astype(np.float64)
        return np.concatenate([X, -1e4 * np.eye(10)])
    return np.repeat(inputs.gaussian_mixture(50, 11, 3, seed=7), 100, axis=0)  # duplicates


@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("kind", ["lattice", "tight", "one_spot", "duplicates"])
def test_hard_inputs(lk, kind):
    X = _hard(kind)
    got = hac.cluster(X, lk, precision=hac.PREC_F32_RECHECK)
    _check(got, hac.cluster(X, lk, precision=hac.PREC_F64), rtol=1e-12)
