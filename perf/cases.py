"""The clustering calls whose speed this library is measured by.

Every case is one call, or one burst of calls, through the public Python
binding (``paper_2106_04727_gb300.hac``), with the options such a program sets.
A case is a dict of plain values:

``entry``      ``run``      a handle made from device points; a pass is
                            ``hac_run`` and ``hac_dendrogram``
               ``cluster``  host points; a pass is ``hac.cluster`` (create, run,
                            dendrogram, destroy), as a script calls it
               ``static``   device points and output; a pass is
                            ``hac_run_static``
               ``batch``    a list of handles; a pass is ``hac_run_batch`` and
                            every handle's ``hac_dendrogram``
               ``serve``    a server that is up; a pass submits a burst of
                            requests, waits for them and polls their results
``data``       shape of the points (the generators below; the recipes are those
               of ``paper_2106_04727_gb300.inputs``, drawn on the GPU)
``n``, ``d``, ``dtype``, ``linkage``, ``f32`` (FP32 bulk with FP64 re-score, or
all FP64), ``slots`` (pair-distance cache), ``count`` (requests of a burst; their
sizes are log-uniform in [64, n]).

A dendrogram comes back in the library's canonical order (height, size, cid)
where heights are FP64 (Ward, avg-2, the all-FP64 mode).  In the FP32 mode
complete and average heights are estimates within 8e-6, whose last bits decide
the order of nearly equal heights; those passes file the merges by the cluster
they retire (each cid but the root retires once), as a program does that cuts
or walks the tree by cluster.
"""
import math

import numpy as np
import torch

from paper_2106_04727_gb300 import hac

EXACT_N = 30_001   # largest n whose FP64 dendrogram exact() builds


def _case(name, entry, data, n, d, linkage, dtype="f32", f32=True, slots=0, count=1):
    return dict(name=name, entry=entry, data=data, n=n, d=d, linkage=linkage, dtype=dtype,
                f32=f32, slots=slots, count=count)


def listed():
    return [
        # the smallest request of the serving stream, as a script's one call:
        # latency, allocations and launches are all of it
        _case("cluster_ward_2d_64", "cluster", "gmm", 64, 2, "ward"),
        # the allocation-free call of a process that owns the GPU's memory, at
        # the 1,024-point FP64 configuration
        _case("static_average_2d_1024", "static", "uniform", 1024, 2, "average", dtype="f64",
              f32=False),
        # an analysis script's default options on a few thousand FP64 points
        _case("run_complete_3d_4999", "run", "gmm", 4999, 3, "complete", dtype="f64", f32=False),
        # many small data sets at once (one engine per kind)
        _case("batch_average_5d_32x4096", "batch", "gmm", 4096, 5, "average", slots=64, count=32),
        # a burst of the serving stream: mixed linkages, dimensions and sizes
        _case("serve_burst_64x65536", "serve", "gmm", 65536, 10, "mixed", slots=64, count=64),
        # an ordinary data set in one call from host memory
        _case("cluster_average_10d_20001", "cluster", "gmm", 20001, 10, "average", slots=128),
        # the all-FP64 mode, for users who want FP64 heights
        _case("run_average_5d_30001_f64", "run", "gmm", 30001, 5, "average", dtype="f64",
              f32=False, slots=128),
        # the benchmark's two runs: 10^6 points of the 5-D mixture
        _case("run_average_5d_1m", "run", "gmm", 1_000_000, 5, "average", slots=128),
        _case("run_ward_5d_1m", "run", "gmm", 1_000_000, 5, "ward"),
        # the paper's GaussianDisc shape under complete linkage
        _case("run_complete_2d_1m", "run", "gaussiandisc", 1_000_000, 2, "complete", slots=128),
        # the largest: 10^7 points of varying density
        _case("run_ward_2d_10m", "run", "spreaders", 10_000_000, 2, "ward"),
        # high dimension with exact ties, where range queries prune little
        _case("run_avg2_16d_150k", "run", "lattice", 150_000, 16, "average_sq"),
    ]


def _log_int(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n))


def _largest(linkage, d, f32, dtype):
    """Largest n a drawn case takes, so that none costs more than the listed ones."""
    if linkage in ("ward", "average_sq"):
        if d <= 3:
            return 4_000_000
        if d <= 8:
            return 1_000_000
        return 150_000 if f32 else 40_000
    if not f32:
        return 30_000 if d <= 8 else 12_000
    if linkage == "average":
        return 1_000_000 if d <= 5 else 300_000 if d <= 8 else 25_000
    return 1_000_000 if d <= 2 else 150_000 if d <= 5 else 20_000


def draw(rng):
    entry = rng.choice(["run", "run", "run", "run", "cluster", "cluster", "static", "batch"])
    d = rng.choice([1, 2, 2, 3, 4, 5, 5, 7, 8, 10, 13, 16])
    linkage = rng.choice(["complete", "average", "average", "ward", "ward", "average_sq"])
    dtype = rng.choice(["f32", "f32", "f64"])
    f32 = rng.random() < 0.7
    data = rng.choice(["gmm", "gmm", "uniform", "gaussiandisc", "spreaders" if d == 2 else "gmm"])
    top = _largest(linkage, d, f32, dtype)
    count = 1
    if entry == "static":
        top = min(top, hac.HAC_STATIC_MAX_N)
    elif entry == "batch":
        top = 4096
        count = rng.randint(4, 40)
    elif entry == "cluster":
        top = min(top, 300_000)
    if entry == "batch":
        n = _log_int(rng, 256, top)
    else:
        n = _log_int(rng, 64, top)
    slots = 0
    if linkage in ("complete", "average") and entry != "static":
        slots = 128 if n > 20_000 else rng.choice([0, 64, 128])
    return dict(entry=entry, data=data, n=n, d=d, linkage=linkage, dtype=dtype, f32=f32,
                slots=slots, count=count)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _points(data, n, d, dtype, seed):
    """Seeded points on the GPU (the recipes of the package's inputs module)."""
    g = _gen(seed)

    def uni(*shape):
        return torch.rand(*shape, device="cuda", dtype=torch.float64, generator=g)

    def nrm(*shape):
        return torch.randn(*shape, device="cuda", dtype=torch.float64, generator=g)

    if data == "gmm":            # 64 isotropic Gaussians in [0, 100]^d (fewer for few points)
        k = max(4, min(64, n // 64))
        c = torch.randint(k, (n,), device="cuda", generator=g)
        x = (100.0 * uni(k, d))[c] + (0.5 + 2.5 * uni(k))[c][:, None] * nrm(n, d)
    elif data == "uniform":      # uniform in a hypergrid of side sqrt(n)
        x = math.sqrt(n) * uni(n, d)
    elif data == "gaussiandisc":  # 90 % in five Gaussians, 10 % uniform noise
        side, m = 5.0 * math.sqrt(n), int(round(0.9 * n))
        x = side * uni(n, d)
        c = torch.arange(m, device="cuda") % 5
        x[:m] = ((side * uni(5, d))[c] + math.sqrt(n) / 6.0 * nrm(m, d)).clamp_(0.0, side)
        x = x[torch.randperm(n, device="cuda", generator=g)]
    elif data == "spreaders":    # reflected random walks of varying step, 1 % noise
        k = max(1, min(200, n // 50))
        per = -(-n // k)
        sig = (1.0 + 49.0 * uni(k))[:, None, None]
        walk = 1e5 * uni(k, 1, d) + torch.cumsum(nrm(k, per, d) * sig, 1)
        walk = torch.remainder(walk, 2e5)
        walk = torch.where(walk > 1e5, 2e5 - walk, walk) + nrm(k, per, d) * sig
        x = walk.reshape(-1, d)[:n]
        x = torch.where(uni(n, 1) < 0.01, 1e5 * uni(n, d), x)
        x = x[torch.randperm(n, device="cuda", generator=g)]
    elif data == "lattice":      # multiples of 2^-8 in [0, 4)^d: exact ties
        x = torch.randint(1024, (n, d), device="cuda", generator=g).double() / 256.0
    else:
        raise ValueError(data)
    return x.to(torch.float32 if dtype == "f32" else torch.float64).contiguous()


def _requests(case, seed):
    """(n, d, linkage, seed) of every request of a batch or burst: the sizes and
    kinds are the case's, the points the seed's."""
    r = np.random.RandomState(case["n"] * 64 + case["count"])
    out = []
    for i in range(case["count"]):
        n = int(round(math.exp(r.uniform(math.log(64), math.log(case["n"])))))
        d, lk = case["d"], case["linkage"]
        if lk == "mixed":
            d, lk = int(r.choice([2, 3, 5, 10])), str(r.choice(["complete", "average", "ward"]))
        out.append((n, d, lk, seed * 1009 + i))
    return out


class _Owner:
    """Handles and servers that live as long as the state that holds them."""

    def __init__(self, destroy):
        self.destroy, self.held = destroy, []

    def take(self, h):
        self.held.append(h)
        return h

    def __del__(self):
        for h in self.held:
            self.destroy(h)


def prepare(case, seed):
    entry, n, d = case["entry"], case["n"], case["d"]
    np_dtype = np.float32 if case["dtype"] == "f32" else np.float64
    prec = hac.PREC_F32_RECHECK if case["f32"] else hac.PREC_F64
    s = dict(entry=entry, n=n, linkage=case["linkage"], prec=prec, slots=case["slots"],
             by_cid=case["f32"] and case["linkage"] in ("complete", "average", "mixed"))

    def handle(n, d, lk, seed):
        x = _points(case["data"], n, d, case["dtype"], seed)
        torch.cuda.synchronize()   # the points are copied on the handle's own stream
        return s["owner"].take(hac.hac_create_device(x.data_ptr(), n, d, np_dtype, lk))

    if entry == "cluster":
        s["x"] = _points(case["data"], n, d, case["dtype"], seed).cpu().numpy()
    elif entry == "static":
        s["x"] = _points(case["data"], n, d, case["dtype"], seed)
        s["out"] = torch.zeros(n - 1, 4, dtype=torch.int64, device="cuda")
        s["dtype"] = np_dtype
        torch.cuda.synchronize()
    elif entry == "run":
        s["owner"] = _Owner(hac.hac_destroy)
        s["h"] = handle(n, d, case["linkage"], seed)
    elif entry == "batch":
        s["owner"] = _Owner(hac.hac_destroy)
        s["sizes"] = [q[0] for q in _requests(case, seed)]
        s["hs"] = [handle(*q) for q in _requests(case, seed)]
    elif entry == "serve":
        s["owner"] = _Owner(hac.hac_server_destroy)
        s["srv"] = s["owner"].take(hac.hac_server_create(1 << 17, precision=prec,
                                                         cache_slots=case["slots"]))
        for dd in (2, 3, 5, 10):   # a server that has been up: its engines exist
            for lk in ("complete", "average", "ward"):
                x = _points(case["data"], 64, dd, case["dtype"], seed + dd).cpu().numpy()
                t = hac.hac_submit(s["srv"], x, lk)
                hac.hac_server_wait(s["srv"], t)
                hac.hac_poll(s["srv"], t, 64)
        s["reqs"] = [(_points(case["data"], q[0], q[1], case["dtype"], q[3]).cpu().numpy(), q[2])
                     for q in _requests(case, seed)]
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _columns(a, b, h, size, by_cid):
    if not by_cid:
        return dict(a=a, b=b, h=h, size=size)
    n = len(a) + 1
    out = dict(a=np.zeros(n, np.int64), h=np.zeros(n), size=np.zeros(n, np.int64))
    out["a"][b], out["h"][b], out["size"][b] = a, h, size
    return out


def _of(m, by_cid):
    return _columns(m["cid_a"], m["cid_b"], m["height"], m["size"], by_cid)


def _joined(parts):
    return {k: np.concatenate([p[k] for p in parts]) for k in parts[0]}


def run(s):
    entry = s["entry"]
    if entry == "run":
        rc = hac.hac_run(s["h"], precision=s["prec"], cache_slots=s["slots"])
        if rc != hac.HAC_OK:
            raise RuntimeError(hac.hac_strerror(rc))
        return _of(hac.hac_dendrogram(s["h"], s["n"]), s["by_cid"])
    if entry == "cluster":
        r = hac.cluster(s["x"], s["linkage"], precision=s["prec"], cache_slots=s["slots"])
        return _columns(r["a"], r["b"], r["h"], r["size"], s["by_cid"])
    if entry == "static":
        x, out = s["x"], s["out"]
        rc = hac.hac_run_static(x.data_ptr(), x.shape[0], x.shape[1], s["dtype"], s["linkage"],
                                out.data_ptr(), len(out), precision=s["prec"],
                                stream=torch.cuda.current_stream().cuda_stream)
        if rc != hac.HAC_OK:
            raise RuntimeError(hac.hac_strerror(rc))
        if not s["by_cid"]:
            return dict(a=out[:, 0], b=out[:, 1], h=out.view(torch.float64)[:, 2],
                        size=out[:, 3])
        m = out.cpu().numpy().view(hac.MERGE_DTYPE).reshape(-1)
        return _of(m, True)
    if entry == "batch":
        rc = hac.hac_run_batch(s["hs"], precision=s["prec"], cache_slots=s["slots"])
        if rc != hac.HAC_OK:
            raise RuntimeError(hac.hac_strerror(rc))
        return _joined([_of(hac.hac_dendrogram(h, n), s["by_cid"])
                        for h, n in zip(s["hs"], s["sizes"])])
    tickets = [hac.hac_submit(s["srv"], x, lk) for x, lk in s["reqs"]]
    parts = []
    for t, (x, lk) in zip(tickets, s["reqs"]):
        hac.hac_server_wait(s["srv"], t)
        rc, m, _ = hac.hac_poll(s["srv"], t, len(x))
        if rc != hac.HAC_OK:
            raise RuntimeError(hac.hac_strerror(rc))
        parts.append(_of(m, True))
    return _joined(parts)


# ---------------------------------------------------------------------------
# what the path cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """The points read once, the merges written once; average linkage needs
    every point pair's distance (each enters exactly one merge's mean), the
    others at least one distance per cluster that ever exists."""
    item = 4 if case["dtype"] == "f32" else 8
    if case["count"] > 1:   # expected sizes of the log-uniform draw
        lo, hi = 64.0, float(case["n"])
        ln = math.log(hi / lo) or 1.0
        n1 = case["count"] * (hi - lo) / ln
        n2 = case["count"] * (hi * hi - lo * lo) / (2.0 * ln)
    else:
        n1, n2 = float(case["n"]), float(case["n"]) ** 2
    d = 5 if case["linkage"] == "mixed" else case["d"]
    pairs = 2.0 * n1
    if case["linkage"] in ("average", "mixed"):
        pairs += (0.5 if case["linkage"] == "average" else 0.5 / 3.0) * n2
    return {"bytes": n1 * d * item + n1 * 32.0, "flops": pairs * (3.0 * d + 2.0)}


def tolerance(case):
    """FP64 heights differ by the rounding and order of FP64 sums.  FP32-mode
    complete and average heights are within 8e-6 of the FP64 value by the
    library's contract (seen between layouts: a few 1e-6).  Merges are those of
    the FP64 tree; two that FP64 rounding cannot tell apart may swap."""
    if case["f32"] and case["linkage"] in ("complete", "average", "mixed"):
        return {"rel": 8e-6, "max": 1.6e-5, "differ": 1e-3}
    return {"rel": 1e-11, "max": 1e-9, "differ": 1e-3}


# ---------------------------------------------------------------------------
# the same dendrogram in 64 bits
# ---------------------------------------------------------------------------

def _dendrogram64(x, linkage):
    """Rounds of merging every reciprocal nearest-neighbour pair of the full
    FP64 matrix, updated by Lance-Williams (complete: max; average and avg-2:
    weighted mean; Ward: its recurrence on squared distances)."""
    x = x.double()
    n = len(x)
    sq = linkage in ("ward", "average_sq")
    D = torch.empty(n, n, dtype=torch.float64, device=x.device)
    step = max(1, (1 << 26) // n)
    for i in range(0, n, step):
        acc = torch.zeros(min(step, n - i), n, dtype=torch.float64, device=x.device)
        for k in range(x.shape[1]):
            t = x[i:i + step, k, None] - x[None, :, k]
            acc += t * t
        D[i:i + step] = acc if sq else acc.sqrt()
    D.fill_diagonal_(math.inf)
    cid = torch.arange(n, device=x.device)
    size = torch.ones(n, dtype=torch.float64, device=x.device)
    ma, mb, mh, ms = [], [], [], []
    while len(cid) > 1:
        K = len(cid)
        nn = torch.empty(K, dtype=torch.long, device=x.device)
        best = torch.empty(K, dtype=torch.float64, device=x.device)
        col = torch.arange(K, device=x.device)
        step = max(1, (1 << 26) // K)
        for i in range(0, K, step):
            r = D[i:i + step]
            m = r.min(1).values
            best[i:i + step] = m
            nn[i:i + step] = torch.where(r == m[:, None], col, K).min(1).values
        i = torch.nonzero((nn[nn] == col) & (col < nn)).flatten()
        j = nn[i]
        ma.append(cid[i])
        mb.append(cid[j])
        mh.append(best[i].sqrt() if linkage == "ward" else best[i])
        ms.append((size[i] + size[j]).long())
        dij = best[i]
        if linkage == "complete":
            D[i] = torch.maximum(D[i], D[j])
            D[:, i] = torch.maximum(D[:, i], D[:, j])
        elif linkage == "ward":
            si, sj = size[i, None], size[j, None]
            D[i] = ((si + size) * D[i] + (sj + size) * D[j] - size * dij[:, None]) / (si + sj + size)
            new = size.clone()
            new[i] += size[j]
            si, sj, nk = size[None, i], size[None, j], new[:, None]
            D[:, i] = ((si + nk) * D[:, i] + (sj + nk) * D[:, j] - nk * dij) / (si + sj + nk)
        else:
            w = (size[i] / (size[i] + size[j]))
            D[i] = w[:, None] * D[i] + (1.0 - w)[:, None] * D[j]
            D[:, i] = w * D[:, i] + (1.0 - w) * D[:, j]
        size[i] += size[j]
        keep = torch.ones(K, dtype=torch.bool, device=x.device)
        keep[j] = False
        k = torch.nonzero(keep).flatten()
        D = D[k][:, k].contiguous()
        D.fill_diagonal_(math.inf)
        cid, size = cid[k], size[k]
    a, b, h, s = (torch.cat(v).cpu().numpy() for v in (ma, mb, mh, ms))
    o = np.lexsort((a, s, h))
    return a[o], b[o], h[o], s[o]


def exact(case, seed):
    if case["entry"] == "serve" or case["n"] > EXACT_N or case["data"] == "lattice":
        return None
    by_cid = case["f32"] and case["linkage"] in ("complete", "average")
    if case["entry"] == "batch":
        return _joined([_columns(*_dendrogram64(_points(case["data"], n, d, case["dtype"], sd),
                                                lk), by_cid)
                        for n, d, lk, sd in _requests(case, seed)])
    x = _points(case["data"], case["n"], case["d"], case["dtype"], seed)
    return _columns(*_dendrogram64(x, case["linkage"]), by_cid)
