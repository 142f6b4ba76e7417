"""The in-warp FP32 evaluation of an average pair, against its stated arithmetic: FP32
partial sums of at most 16 distances, added in FP64, the mean rounded to FP32 once.
All distances between the clusters are the same FP32 number s, which is read off a
pair whose mean it is."""
import numpy as np
import pytest

from paper_2106_04727_gb300 import hac

pytestmark = pytest.mark.gpu

F = np.float32


def _chunk(s, n):
    t = F(0)
    for _ in range(n):
        t = F(t + s)
    return float(t)


@pytest.mark.parametrize("p", [1.003, 1.1, 1.9])
def test_large_pairs(p, monkeypatch):
    """36 * 10^6 point pairs in one warp (no cache): 70,688 partial sums a lane, all
    equal (offsets too small to change a distance), so the mean is a sixteenth of
    one.  Their rounding errors, all on one side, must not add up."""
    monkeypatch.setenv("HAC_DENSE_K", "0")
    p, m = F(p), 6016
    r = np.random.RandomState(9)

    def line(n, x):   # n points within 2^-18 of (x, 0)
        return np.stack([np.full(n, x, F), (r.uniform(size=n) * 2.0**-18).astype(F)], 1)

    def top(a, b):
        X = np.concatenate([line(a, F(0)), line(b, p)])
        return hac.cluster(X, "average", precision=hac.PREC_F32_RECHECK)["h"][-1]

    c = F(5.9604645e-8)
    up = F(1) + ((F(2) + F(16)) * c + F(32) * c)   # heights are the estimate's upper bound
    one = top(64, 1)
    s = [x for x in (F(p + k * np.spacing(p)) for k in range(-3, 4)) if F(x * up) == F(one)]
    assert s
    assert top(m, m) in [float(F(F(_chunk(x, 16) / 16.0) * up)) for x in s]
