"""Inputs far from unit scale.  Coordinates times 2^k give the same merges in the
same rounds with heights times 2^k (avg-2: 4^k), bit for bit in the FP64 mode,
through every entry point: the bounds that steer the searches are FP32, and a
search whose bounds are all infinite must neither lose its neighbour nor run on."""
import numpy as np
import pytest

import oracle
from paper_2106_04727_gb300 import hac, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LKS = ["complete", "average", "ward", "average_sq"]


def _slots(prec):  # cached FP64 sums depend on which pairs were evaluated before
    return 32 if prec == hac.PREC_F32_RECHECK else 0


def _static(X, lk, prec):
    n, d = X.shape
    src = torch.from_numpy(X).cuda()
    out = torch.zeros((n - 1) * 4, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    rc = hac.hac_run_static(src.data_ptr(), n, d, X.dtype, lk, out.data_ptr(), n - 1, precision=prec)
    assert rc == hac.HAC_OK
    return hac.result_dict(out.cpu().numpy().view(hac.MERGE_DTYPE))


def _batch(X, lk, prec):
    hs = [hac.hac_create(X, lk), hac.hac_create(np.ascontiguousarray(X[::2]), lk)]
    try:
        assert hac.hac_run_batch(hs, precision=prec, cache_slots=_slots(prec)) == hac.HAC_OK
        return hac.result_dict(hac.hac_dendrogram(hs[0], len(X)))
    finally:
        for h in hs:
            hac.hac_destroy(h)


CALLS = {"run": lambda X, lk, prec: hac.cluster(X, lk, precision=prec, cache_slots=32),
         "tree": lambda X, lk, prec: hac.cluster(X, lk, precision=prec, cache_slots=_slots(prec),
                                                 timeout_s=60.0),
         "static": _static, "batch": _batch}


# 2^100: FP32 squares overflow; 2^200: FP32 itself; 2^900: FP64 squares; and below
@pytest.mark.parametrize("entry", list(CALLS))
@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("k", [-900, -200, -100, -60, 47, 70, 100, 200, 900])
def test_fp64_scales_exactly(lk, entry, k, monkeypatch):
    if entry == "tree":
        monkeypatch.setenv("HAC_DENSE_K", "0")
    X = inputs.gaussian_mixture(330, 3, 5, seed=17, dtype=np.float64)
    want = oracle.nnchain(X, lk)
    one = CALLS[entry](X, lk, hac.PREC_F64)
    c = oracle.compare(one, want, rtol=1e-9)
    assert c["ok"], c
    got = CALLS[entry](np.ldexp(X, k), lk, hac.PREC_F64)
    order = lambda t: np.argsort(t["b"])
    a, b = order(one), order(got)
    for f in ("a", "b", "size"):
        assert np.array_equal(one[f][a], got[f][b])
    with np.errstate(over="ignore", under="ignore"):
        assert np.array_equal(np.ldexp(one["h"][a], 2 * k if lk == "average_sq" else k),
                              got["h"][b])


@pytest.mark.parametrize("entry", list(CALLS))
@pytest.mark.parametrize("lk", LKS)
@pytest.mark.parametrize("k", [-100, -70, 100])
@pytest.mark.parametrize("dt", [np.float32, np.float64])
def test_fp32_mode(lk, entry, k, dt, monkeypatch):
    if entry == "tree":
        monkeypatch.setenv("HAC_DENSE_K", "0")
    X = inputs.gaussian_mixture(330, 3, 5, seed=18, dtype=dt)
    if entry == "batch" and k > 0:  # an FP32 batch refuses coordinates of 2^40 or more
        h = hac.hac_create(np.ldexp(X, k), lk)
        try:
            assert hac.hac_run_batch([h], precision=hac.PREC_F32_RECHECK) == hac.HAC_EINVAL
        finally:
            hac.hac_destroy(h)
        return
    got = CALLS[entry](np.ldexp(X, k), lk, hac.PREC_F32_RECHECK)
    with np.errstate(over="ignore", under="ignore"):
        got["h"] = np.ldexp(got["h"], -2 * k if lk == "average_sq" else -k)
    c = oracle.compare(got, oracle.nnchain(X.astype(np.float64), lk), rtol=1e-5)
    assert c["ok"], c


@pytest.mark.parametrize("entry", list(CALLS))
@pytest.mark.parametrize("lk", LKS)
def test_next_to_the_largest_number(lk, entry, monkeypatch):
    """All coordinates near 1.5 * 10^308: the sum of the box's ends is beyond FP64."""
    if entry == "tree":
        monkeypatch.setenv("HAC_DENSE_K", "0")
    Y = inputs.gaussian_mixture(300, 2, 4, seed=19, dtype=np.float64)
    X = np.ldexp(Y, 1010) + 1.5e308
    Y = np.ldexp(X, -1010) - np.ldexp(1.5e308, -1010)   # the same points, exactly
    got = CALLS[entry](X, lk, hac.PREC_F64)
    want = oracle.nnchain(Y, lk)
    if lk == "average_sq":   # heights are beyond FP64: the merges by size and order
        assert np.all(np.isinf(got["h"][want["h"] > 1e-3]))
        assert sorted(zip(got["a"], got["b"])) == sorted(zip(want["a"], want["b"]))
        return
    got["h"] = np.ldexp(got["h"], -1010)
    c = oracle.compare(got, want, rtol=1e-9)
    assert c["ok"], c
