"""Average linkage: exactly tied means are decided by cid, whichever way round the two
clusters lie in the matrix, and whatever their sizes."""
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


def _exact(x):
    """Algorithm 1 on integers on a line, means compared as fractions."""
    n = len(x)
    S = [[abs(a - b) for b in x] for a in x]
    size, act, succ, out = [1] * n, list(range(n)), {}, []
    while len(act) > 1:
        new = {}
        for i in act:
            if i not in succ:
                best = None
                for j in act:   # sum / (|i| |j|): |i| is common
                    if j != i and (best is None or S[i][j] * size[best] < S[i][best] * size[j]):
                        best = j
                new[i] = best
        succ.update(new)
        pairs = [(i, succ[i]) for i in act if i < succ[i] and succ[succ[i]] == i]
        for i, j in pairs:
            out.append((i, j, size[i] + size[j]))
            size[i] += size[j]
            for k in range(n):
                S[i][k] += S[j][k]
            for k in range(n):
                S[k][i] += S[k][j]
        gone = {j for _, j in pairs}
        touched = gone | {i for i, _ in pairs}
        act = [i for i in act if i not in gone]
        succ = {i: j for i, j in succ.items() if i not in touched and j not in touched}
    return sorted(out)


@pytest.mark.parametrize("call", list(CALLS))
def test_integers_on_a_line(call):
    """Many true ties between clusters of different sizes."""
    for seed in range(12):
        r = np.random.RandomState(seed)
        x = r.randint(0, r.choice([40, 100, 400]), r.randint(60, 180))
        got = CALLS[call](x.astype(np.float64)[:, None])
        assert sorted(zip(got["a"], got["b"], got["size"])) == _exact(x.tolist()), seed
