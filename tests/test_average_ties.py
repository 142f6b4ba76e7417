"""Average linkage: exactly tied means are decided by cid, whichever way round the two
clusters lie in the matrix."""
import numpy as np
import pytest

from paper_2106_04727_gb300 import hac

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _static(X):
    n, d = X.shape
    src = torch.from_numpy(X).cuda()
    out = torch.zeros((n - 1) * 4, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert hac.hac_run_static(src.data_ptr(), n, d, X.dtype, "average", out.data_ptr(),
                              n - 1) == hac.HAC_OK
    return hac.result_dict(out.cpu().numpy().view(hac.MERGE_DTYPE))


CALLS = {"f64": lambda X: hac.cluster(X, "average"),
         "f32recheck": lambda X: hac.cluster(X, "average", precision=hac.PREC_F32_RECHECK),
         "static": _static}


@pytest.mark.parametrize("call", list(CALLS))
@pytest.mark.parametrize("sizes", [(3, 5), (5, 3), (3, 7), (7, 10), (11, 6)])
def test_mirror_images(sizes, call):
    """A symmetric cluster of `mid` points between two mirror images of `side` points,
    one first and one last in the input: equal sums and sizes, so the middle joins
    the first."""
    mid, side = sizes
    for trial in range(40):
        r = np.random.RandomState(100 * mid + side + 1000 * trial)
        half = r.choice(np.arange(1, 40), mid // 2, replace=False)
        m = np.concatenate([half, -half, [0] * (mid % 2)])
        s = r.randint(3000, 4000) + r.choice(np.arange(60), side, replace=False)
        X = np.concatenate([-s, m, s]).astype(np.float64)[:, None]
        got = CALLS[call](X)
        pairs = {(int(a), int(b)): int(z) for a, b, z in zip(got["a"], got["b"], got["size"])}
        assert pairs.get((0, side)) == mid + side, trial
