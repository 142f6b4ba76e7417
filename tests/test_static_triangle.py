"""hac_run_static's FP64 rounds on the packed triangle (csrc/hac_dense.cu) and
the one-block record sort: sizes around the triangle's capacity, its 64- and
200-cluster block counts, exact ties, and the calls that stay on the ordinary
rounds."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2106_04727_gb300 import hac, inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _static(X, lk, **opts):
    n, d = X.shape
    src = torch.from_numpy(X).cuda()
    out = torch.zeros((n - 1) * 4, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    o = hac.hac_default_opts()
    for k, v in opts.items():
        setattr(o, k, v)
    rc = hac.load().hac_run_static(src.data_ptr(), n, d, hac.F32 if X.dtype == np.float32 else hac.F64,
                                   hac.LINKAGES[lk], ctypes.byref(o), out.data_ptr(), n - 1)
    m = out.cpu().numpy().view(hac.MERGE_DTYPE)
    return rc, dict(a=m["cid_a"], b=m["cid_b"], h=m["height"], size=m["size"])


# from the points (2-D: 1,100 clusters fit), and after ordinary rounds
@pytest.mark.parametrize("lk", ["complete", "average"])
@pytest.mark.parametrize("n,d,dt", [(2, 2, np.float64), (33, 1, np.float32), (65, 5, np.float64),
                                    (201, 16, np.float32), (1024, 2, np.float64),
                                    (1281, 2, np.float32), (1500, 9, np.float64),
                                    (4096, 16, np.float32), (4096, 3, np.float64)])
def test_sizes(lk, n, d, dt):
    X = inputs.gaussian_mixture(n, d, 6, seed=n + d, dtype=dt)
    rc, got = _static(X, lk)
    assert rc == hac.HAC_OK
    c = oracle.compare(got, oracle.nnchain(X.astype(np.float64), lk), rtol=1e-9)
    assert c["ok"], c
    order = np.lexsort((got["a"], got["size"], got["h"]))
    assert np.array_equal(order, np.arange(n - 1))


@pytest.mark.parametrize("lk", ["complete", "average"])
def test_ties(lk):
    X = inputs.lattice(700, 2, seed=8, levels=9).astype(np.float64)
    rc, got = _static(X, lk)
    assert rc == hac.HAC_OK
    bad, stats = oracle.validate(X, lk, got, rtol=1e-9, htol=1e-9)
    assert bad == 0, stats


@pytest.mark.parametrize("lk", ["complete", "average"])
def test_limits_and_no_prune(lk):
    X = inputs.gaussian_mixture(900, 2, 5, seed=4, dtype=np.float64)
    want = oracle.nnchain(X, lk)
    assert _static(X, lk, max_rounds=3)[0] == hac.HAC_ETIMEOUT
    for opts in (dict(timeout_s=60.0), dict(flags=hac.HAC_FLAG_NO_PRUNE), {}):
        rc, got = _static(X, lk, **opts)
        assert rc == hac.HAC_OK and oracle.compare(got, want, rtol=1e-9)["ok"]
    Y = X.copy()
    Y[5, 1] = np.inf
    assert _static(Y, lk)[0] == hac.HAC_EINVAL


@pytest.mark.parametrize("lk", ["complete", "average"])
@pytest.mark.parametrize("n,d,levels", [(201, 3, 9), (201, 5, 4), (700, 8, 4), (900, 2, 9),
                                        (1100, 2, 40), (1280, 1, 500)])
def test_ties_as_on_the_matrix(lk, n, d, levels):
    """Exact sums: lattice points' many tied distances give the tree and the heights of
    hac_run's matrix bit for bit, whatever limits the call carries."""
    X = inputs.lattice(n, d, seed=n, levels=levels).astype(np.float64)
    want = hac.cluster(X, lk)
    assert want["stats"]["dense_k"] == n
    for opts in ({}, dict(timeout_s=60.0), dict(max_rounds=n)):
        rc, got = _static(X, lk, **opts)
        assert rc == hac.HAC_OK
        for f in ("a", "b", "h", "size"):
            assert np.array_equal(got[f], want[f]), (f, opts)
