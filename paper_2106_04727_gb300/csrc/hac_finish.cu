// The last rounds of a closed-form linkage (Ward, avg-2) in one launch.
//
// Once few clusters are active a round of Algorithm 1 is all latency: about
// 15 launches and two host reads for microseconds of work (85-110 us a round
// measured at K <= 2,048).  Here one thread-block cluster (up to 16 SMs) runs
// every remaining round: the active clusters' FP32 records sit whole in every
// block's shared memory, a warp scans them all for one terminal (no tree),
// and the phases of a round (search; FP64 keys and chain update; reciprocal
// filter and merges; compaction) are separated by the hardware cluster
// barrier instead of launches.  Rounds, pairs and merge records are those of
// round_step: the search returns the candidate of least (FP64 key, cid), and
// keys, sums and centroids are computed by the same FP64 expressions.
//
// What bounds it: latency (three or four cluster barriers and the dependent L2
// reads of each phase, about 10 us a round at K <= 256), and above K = 1,000
// the scans' FP32 issue (16 SMs; K = 3,805 to the end, 5-D Ward: 1.14 ms for
// 34 rounds that took 3.6 ms).
//
// Screening.  FP32 distances only exclude candidates: with the error model of
// hac_query.cuh (|D32 - D| <= delta + rho D, delta = 2.01 u M sqrt(d)
// [* sqrt(w) for Ward]), U = least upper bound; a terminal whose second least
// lower bound exceeds U has its winner, any other re-scores every candidate
// within U in FP64.  The coordinates' scale (unit_exp) keeps the FP32 squares from
// overflow and flush; inputs without one (all points equal, subnormal extent) take
// the ordinary rounds.
//
// "Direct" runs (n within the capacity) start from the input points: bounding
// box, recentring and the singletons' state are made by the same kernel, and
// it writes the dendrogram in canonical order itself, so a whole hac_run is
// one launch.  Both the spatial order and the tree only steer pruning, so
// leaving them out does not change a merge.
#include "hac_impl.cuh"

#include <algorithm>
#include <cmath>

namespace hacg {

namespace {

constexpr int FT = 1024;              // threads of a block
constexpr int FW = FT / 32;
constexpr int FIN_PER = FIN_MAX_K / FT;  // list entries per thread in the compaction
constexpr float FU32 = 5.9604645e-8f;    // 2^-24

__device__ __forceinline__ int cta_rank() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ int cta_count() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// all threads of the cluster: what was written before is read after (reads of
// data another block writes go to L2, __ldcg)
__device__ __forceinline__ void cluster_sync_all() {
  __threadfence();
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// exclusive scan over the block's FT threads of two counts packed in one int
// (low and high 16 bits; each total is at most FIN_MAX_K)
__device__ int fin_scan(int v, int *total, int *ws) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    int t = ws[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    ws[lane] = t;
  }
  __syncthreads();
  const int pre = w ? ws[w - 1] : 0;
  *total = ws[FW - 1];
  __syncthreads();
  return pre + x - v;
}

// FP64 key of (A = i, B = j), as the search of hac_query.cuh computes it
template <int LK, int D>
__device__ double closed_key(const State &s, int i, int j) {
  const int dp = s.dp;
  const int na = __ldcg(&s.csize[i]), nb = __ldcg(&s.csize[j]);
  double g2 = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    if (k < s.d) {
      const double t = __ldcg(&s.cent[(size_t)i * dp + k]) - __ldcg(&s.cent[(size_t)j * dp + k]);
      g2 += t * t;
    }
  }
  if (LK == LK_AVG2)
    return g2 + __ldcg(&s.sse[i]) / (double)na + __ldcg(&s.sse[j]) / (double)nb;
  return (2.0 * (double)na * (double)nb) / (double)(na + nb) * g2;
}

// records of this round's active clusters, one copy per block
struct FinSm {
  float *x;    // coordinate k of cluster p at x[k * Kc + p]
  float *g;    // Ward: 1 / size; avg-2: variance (SSE / size)
  int *cid;    // active cids in order
  int *term;   // positions of the terminals
};

template <int LK, int D>
__device__ __forceinline__ void fin_gather(const State &s, const FinSm &m, int Kc, int K) {
  const int dp = s.dp;
  for (int p = threadIdx.x; p < K; p += FT) {
    const int c = m.cid[p];
#pragma unroll
    for (int k = 0; k < D; ++k)
      m.x[k * Kc + p] = k < s.d ? __ldcg(&s.cent32[(size_t)c * dp + k]) : 0.f;
    const int sz = __ldcg(&s.csize[c]);
    m.g[p] = LK == LK_WARD ? 1.f / (float)sz
                           : (sz > 1 ? (float)(__ldcg(&s.sse[c]) / (double)sz) : 0.f);
  }
}

// Bounds of candidate p for a terminal: `lo` and `up` on D^2 (Ward, up to
// (1 -/+ rho)^2) or on D = sqrt(key) (avg-2, up to 1 -/+ rho).
template <int LK, int D>
__device__ __forceinline__ void fin_bounds(const FinSm &m, int Kc, int p, const float (&c)[D],
                                           float ga, float delta, float &lo, float &up) {
  float dc2 = 0.f;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float t = c[k] - m.x[k * Kc + p];
    dc2 = fmaf(t, t, dc2);
  }
  const float gb = m.g[p];
  if (LK == LK_WARD) {
    const float w = 2.f * rcp_approx(ga + gb);  // 2|A||B| / (|A| + |B|)
    const float sd = sqrt_approx_ftz(dc2);
    const float a = fmaxf(sd - delta, 0.f), b = sd + delta;
    lo = w * a * a;
    up = w * b * b;
  } else {
    const float sd = sqrt_approx_ftz(dc2 + ga + gb);
    lo = fmaxf(sd - delta, 0.f);
    up = sd + delta;
  }
}

// One terminal by one warp: its nearest neighbour into Ecid, with the FP64 key
// in Ekey if it was needed to decide (else -1: the key follows in fin_keys).
template <int LK, int D>
__device__ void fin_search(const State &s, const FinSm &m, int Kc, int K, int self, float delta,
                           float rho2, int lane, int &evals) {
  float c[D];
#pragma unroll
  for (int k = 0; k < D; ++k) c[k] = m.x[k * Kc + self];
  const float ga = m.g[self];
  float L1 = INFINITY, L2 = INFINITY, U = INFINITY;
  int p1 = -1;
#pragma unroll 2
  for (int p = lane; p < K; p += 32) {
    float lo, up;
    fin_bounds<LK, D>(m, Kc, p, c, ga, delta, lo, up);
    if (p == self) lo = up = INFINITY;
    if (lo < L1) {
      L2 = L1;
      L1 = lo;
      p1 = p;
    } else {
      L2 = fminf(L2, lo);
    }
    U = fminf(U, up);
  }
  float l1 = L1, u = U;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    l1 = fminf(l1, __shfl_xor_sync(0xffffffffu, l1, o));
    u = fminf(u, __shfl_xor_sync(0xffffffffu, u, o));
  }
  const float lim = u * (1.f + rho2);
  // candidates that can be the FP64 winner: lo (1 - rho2) <= lim
  const unsigned first = __ballot_sync(0xffffffffu, L1 * (1.f - rho2) <= lim);
  const unsigned second = __ballot_sync(0xffffffffu, L2 * (1.f - rho2) <= lim);
  const int ci = m.cid[self];
  if (__popc(first) == 1 && !second) {
    const int p = __shfl_sync(0xffffffffu, p1, __ffs(first) - 1);
    if (lane == 0) {
      s.Ecid[ci] = m.cid[p];
      s.Ekey[ci] = -1.0;
    }
    return;
  }
  unsigned long long bk = ~0ull;
  int bc = INT_MAX;
  for (int p = lane; p < K; p += 32) {
    float lo, up;
    fin_bounds<LK, D>(m, Kc, p, c, ga, delta, lo, up);
    if (p == self || !(lo * (1.f - rho2) <= lim)) continue;
    ++evals;
    const int cb = m.cid[p];
    const unsigned long long k =
        (unsigned long long)__double_as_longlong(closed_key<LK, D>(s, ci, cb));
    if (k < bk || (k == bk && cb < bc)) {
      bk = k;
      bc = cb;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, bk, o);
    const int c2 = __shfl_xor_sync(0xffffffffu, bc, o);
    if (k2 < bk || (k2 == bk && c2 < bc)) {
      bk = k2;
      bc = c2;
    }
  }
  if (lane == 0) {
    s.Ecid[ci] = bc == INT_MAX ? -1 : bc;
    s.Ekey[ci] = __longlong_as_double((long long)bk);
    if (bc == INT_MAX) atomicOr(&s.ctr->err, ERR_NO_NN);
  }
}

// a reciprocal pair becomes one cluster: the expressions of k_merge
template <int D>
__device__ void fin_merge(const State &s, int i, int j, int round) {
  const int lo = min(i, j), hi = max(i, j), dp = s.dp;
  const double key = __ldcg(&s.Ekey[i]);
  const int na = __ldcg(&s.csize[lo]), nb = __ldcg(&s.csize[hi]);
  const int r = s.irec[0] + atomicAdd(&s.irecn[0], 1);
  s.m_a[r] = lo;
  s.m_b[r] = hi;
  s.m_h[r] = s.linkage == LK_WARD ? sqrt(key) : key;
  s.m_size[r] = na + nb;
  s.m_round[r] = round;
  const double inv = 1.0 / (double)(na + nb);
  double g2 = 0.0;
#pragma unroll
  for (int k = 0; k < D; ++k)
    if (k < s.d) {
      const double t = __ldcg(&s.cent[(size_t)lo * dp + k]) - __ldcg(&s.cent[(size_t)hi * dp + k]);
      g2 += t * t;
    }
  s.sse[lo] = __ldcg(&s.sse[lo]) + __ldcg(&s.sse[hi]) + (double)na * (double)nb * inv * g2;
#pragma unroll
  for (int k = 0; k < D; ++k)
    if (k < s.d) {
      const double sum = __ldcg(&s.csum[(size_t)lo * dp + k]) + __ldcg(&s.csum[(size_t)hi * dp + k]);
      s.csum[(size_t)lo * dp + k] = sum;
      const double c = sum * inv;
      s.cent[(size_t)lo * dp + k] = c;
      s.cent32[(size_t)lo * dp + k] = (float)c;
    }
  s.csize[lo] = na + nb;
  s.succ[lo] = -1;
  s.mround[lo] = round;
  s.mround[hi] = round;
  s.alive[hi] = 0;
}

// Direct runs: bounding box, recentring and the singletons' state.  Returns
// false when the input is not for this path (non-finite, or a scale the FP32
// screening does not take); uniform over the cluster.
template <typename T, int LK, int D>
__device__ bool fin_start(const FinArgs &a, const FinSm &m, double *s_box, float *scale_out) {
  const State &s = a.s;
  const T *X = (const T *)a.raw;
  const int n = a.K, d = s.d, dp = s.dp;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __shared__ int s_bad;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  if (w < d) {  // one warp per coordinate
    double lo = INFINITY, hi = -INFINITY;
    bool bad = false;
    for (int i = lane; i < n; i += 32) {
      const double x = (double)X[(size_t)i * d + w];
      if (!isfinite(x)) bad = true;
      lo = fmin(lo, x);
      hi = fmax(hi, x);
    }
    for (int o = 16; o; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (__any_sync(0xffffffffu, bad)) s_bad = 1;
    if (lane == 0) {
      s_box[w] = lo;
      s_box[MAXD + w] = hi;
    }
  }
  __syncthreads();
  if (s_bad) {
    if (cta_rank() == 0 && threadIdx.x == 0) atomicOr(&s.ctr->err, ERR_NONFINITE);
    return false;
  }
  double scale = 0.0;
  for (int k = 0; k < d; ++k) {
    const double c = box_centre(s_box[k], s_box[MAXD + k]);
    scale = fmax(scale, fmax(fabs(s_box[k] - c), fabs(s_box[MAXD + k] - c)));
  }
  const int ue = unit_exp(scale);
  const double mul = ldexp(1.0, -ue);
  scale *= mul;
  if (!(scale >= FIN_SCALE_LO && scale < FIN_SCALE_HI)) {  // all points equal, or subnormal
    if (cta_rank() == 0 && threadIdx.x == 0) s.ctr->fin_refused = 1;
    return false;
  }
  *scale_out = (float)(scale * (1.0 + 1e-6));
  for (int i = threadIdx.x; i < n; i += FT) {
    m.cid[i] = i;
    m.term[i] = i;
    m.g[i] = LK == LK_WARD ? 1.f : 0.f;
#pragma unroll
    for (int k = 0; k < D; ++k)
      m.x[k * a.Kc + i] =
          k < d ? (float)(((double)X[(size_t)i * d + k] - box_centre(s_box[k], s_box[MAXD + k])) * mul)
                : 0.f;
  }
  for (int i = cta_rank() * FT + threadIdx.x; i < n; i += cta_count() * FT) {
    for (int k = 0; k < d; ++k) {
      const double x = ((double)X[(size_t)i * d + k] - box_centre(s_box[k], s_box[MAXD + k])) * mul;
      s.csum[(size_t)i * dp + k] = x;
      s.cent[(size_t)i * dp + k] = x;
      s.cent32[(size_t)i * dp + k] = (float)x;
    }
    s.sse[i] = 0.0;
    s.csize[i] = 1;
    s.succ[i] = -1;
    s.mround[i] = -1;
    s.isterm[i] = 0;
    s.alive[i] = 1;
  }
  if (cta_rank() == 0 && threadIdx.x == 0) {
    s.irec[0] = 0;
    s.irecn[0] = 0;
    s.iunit[0] = ldexp(1.0, ue);
  }
  return true;
}

// The canonical order (height, size, cid_a) of a direct run's m records, by a
// bitonic sort in the shared memory of one block.
__device__ void fin_records(const State &s, int m, hac_merge *out, int32_t *out_round,
                            unsigned char *smem) {
  int P = 32;
  while (P < m) P <<= 1;
  unsigned long long *kh = (unsigned long long *)smem;
  unsigned long long *ks = kh + P;
  int *idx = (int *)(ks + P);
  for (int i = threadIdx.x; i < P; i += FT) {
    const bool v = i < m;
    kh[i] = v ? (unsigned long long)__double_as_longlong(__ldcg(&s.m_h[i])) : ~0ull;
    ks[i] = v ? ((unsigned long long)(unsigned)__ldcg(&s.m_size[i]) << 32) |
                    (unsigned)__ldcg(&s.m_a[i])
              : ~0ull;
    idx[i] = i;
  }
  __syncthreads();
  for (int len = 2; len <= P; len <<= 1)
    for (int st = len >> 1; st; st >>= 1) {
      for (int q = threadIdx.x; q < P / 2; q += FT) {
        const int i = ((q & ~(st - 1)) << 1) | (q & (st - 1)), j = i | st;
        const bool asc = (i & len) == 0;
        const unsigned long long hi = kh[i], hj = kh[j], si = ks[i], sj = ks[j];
        const bool gt = hi > hj || (hi == hj && si > sj);
        const bool lt = hi < hj || (hi == hj && si < sj);
        if (asc ? gt : lt) {
          kh[i] = hj;
          kh[j] = hi;
          ks[i] = sj;
          ks[j] = si;
          const int t = idx[i];
          idx[i] = idx[j];
          idx[j] = t;
        }
      }
      __syncthreads();
    }
  const double unit = __ldcg(s.iunit);
  for (int i = threadIdx.x; i < m; i += FT) {
    const int v = idx[i];
    hac_merge r;
    r.cid_a = (int)(unsigned)ks[i];
    r.cid_b = __ldcg(&s.m_b[v]);
    r.height = unit_height(__longlong_as_double((long long)kh[i]), unit, s.linkage == LK_AVG2);
    r.size = (int)(ks[i] >> 32);
    out[i] = r;
    out_round[i] = __ldcg(&s.m_round[v]);
  }
}

template <int LK, int D>
__global__ void __launch_bounds__(FT, 1) k_finish(FinArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int ws[FW];
  __shared__ double s_box[2 * MAXD];
  const State &s = a.s;
  const int Kc = a.Kc;
  FinSm m;
  m.x = (float *)smem;
  m.g = m.x + (size_t)D * Kc;
  m.cid = (int *)(m.g + Kc);
  m.term = m.cid + Kc;
  const int rank = cta_rank(), nct = cta_count();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int K = a.K, nterm = a.nterm, round = a.round;
  float scale = a.scale;
  if (a.raw) {
    const bool ok = a.in_f32 ? fin_start<float, LK, D>(a, m, s_box, &scale)
                             : fin_start<double, LK, D>(a, m, s_box, &scale);
    if (!ok) return;  // every block of the cluster took the same decision
  } else {
    for (int p = threadIdx.x; p < K; p += FT) m.cid[p] = a.order[p];
    for (int t = threadIdx.x; t < nterm; t += FT) m.term[t] = s.pos[s.term[t]];
    __syncthreads();
    fin_gather<LK, D>(s, m, Kc, K);
  }
  cluster_sync_all();
  const float delta = 2.01f * FU32 * scale * sqrtf((float)s.d) * 1.01f;
  // (1 -/+ rho)^2 of the squared bounds (Ward); a little more than needed for avg-2
  const float rho2 = 2.2f * ((float)s.d + 16.f) * FU32;
  long long searches = 0, naive = 0;
  int evals = 0;
  const int round_end = a.rounds_max > 0 ? round + a.rounds_max : INT_MAX;
  while (K > 1 && round < round_end) {
    searches += nterm;
    naive += (long long)nterm * (K - 1);
    for (int t = rank * FW + wid; t < nterm; t += nct * FW)
      fin_search<LK, D>(s, m, Kc, K, m.term[t], delta, rho2, lane, evals);
    cluster_sync_all();
    // FP64 keys of the decided terminals, chain update
    for (int t = rank * FT + threadIdx.x; t < nterm; t += nct * FT) {
      const int i = m.cid[m.term[t]];
      const int j = __ldcg(&s.Ecid[i]);
      if (j < 0) continue;
      if (__ldcg(&s.Ekey[i]) < 0.0) {
        s.Ekey[i] = closed_key<LK, D>(s, i, j);
        ++evals;
      }
      s.succ[i] = j;
    }
    cluster_sync_all();
    // reciprocal pairs merge, each by one thread (a thread that reads succ of
    // a cluster merging meanwhile sees its partner or -1: no match either way)
    for (int t = rank * FT + threadIdx.x; t < nterm; t += nct * FT) {
      const int i = m.cid[m.term[t]];
      const int j = __ldcg(&s.Ecid[i]);
      if (j < 0) continue;
      if (__ldcg(&s.succ[j]) == i && (i < j || __ldcg(&s.isterm[j]) != round))
        fin_merge<D>(s, i, j, round);
    }
    cluster_sync_all();
    // chain repair and stable compaction, the same in every block
    int c[FIN_PER], f[FIN_PER], cnt = 0;
#pragma unroll
    for (int r = 0; r < FIN_PER; ++r) {
      const int p = threadIdx.x * FIN_PER + r;
      c[r] = p < K ? m.cid[p] : -1;
      f[r] = 0;
      if (c[r] >= 0 && __ldcg(&s.alive[c[r]])) {
        int sc = __ldcg(&s.succ[c[r]]);
        if (sc >= 0 && __ldcg(&s.mround[sc]) == round) {
          sc = -1;
          if (rank == 0) s.succ[c[r]] = -1;
        }
        f[r] = 1 | (sc < 0 ? 1 << 16 : 0);
      }
      cnt += f[r];
    }
    int tot;
    int at = fin_scan(cnt, &tot, ws);
    const int K2 = tot & 0xffff;
    if (K2 >= K) {  // no pair merged: cannot happen
      if (rank == 0 && threadIdx.x == 0) atomicOr(&s.ctr->err, ERR_NO_NN);
      break;
    }
#pragma unroll
    for (int r = 0; r < FIN_PER; ++r) {
      if (f[r]) {
        m.cid[at & 0xffff] = c[r];
        if (f[r] >> 16) {
          m.term[at >> 16] = at & 0xffff;
          if (rank == 0) s.isterm[c[r]] = round + 1;
        }
      }
      at += f[r];
    }
    __syncthreads();
    K = K2;
    nterm = tot >> 16;
    ++round;
    fin_gather<LK, D>(s, m, Kc, K);
    __syncthreads();
  }
  evals = __reduce_add_sync(0xffffffffu, evals);
  if (lane == 0 && evals) atomicAdd(&s.ctr->cluster_pairs, (unsigned long long)evals);
  if (rank != 0) return;
  if (threadIdx.x == 0) {
    s.ctr->nactive = K;
    s.ctr->nterm = nterm;
    s.ctr->nmerges += a.K - K;
    s.ctr->ltests += (unsigned long long)naive;
    s.ctr->fin_rounds = round - a.round;
    s.ctr->fin_searches = searches;
    s.ctr->fin_naive = naive;
    if (K <= 1) s.idone[0] = 1;
    s.iact[0] = K;
  }
  if (K > 1) {  // stopped by the round limit: the lists go back
    for (int p = threadIdx.x; p < K; p += FT) {
      a.order_out[p] = m.cid[p];
      s.pos[m.cid[p]] = p;
    }
    for (int t = threadIdx.x; t < nterm; t += FT) s.term[t] = m.cid[m.term[t]];
  } else if (a.out) {
    __syncthreads();
    fin_records(s, a.n_rec, a.out, a.out_round, smem);
  }
}

// The same for the records of any run: at most FIN_MAX_K of them sort faster in
// one block than by 14 grid-wide radix passes of 5 launches (whole 2-D average
// runs of 64 and 1,024 points: 0.70 and 1.06 ms before, 0.27 and 0.56 with this
// and without the spatial sort that no tree search follows).
__global__ void __launch_bounds__(FT, 1) k_rec_sort(State s, int m, hac_merge *out,
                                                    int32_t *out_round) {
  extern __shared__ __align__(16) unsigned char smem[];
  fin_records(s, m, out, out_round, smem);
}

int fin_pow2(int m) {
  int P = 32;
  while (P < m) P <<= 1;
  return P;
}
constexpr int REC_BYTES = 20;  // sorted per record
constexpr int FIN_REC_SMEM = FIN_MAX_K * REC_BYTES;
static_assert(FIN_REC_SMEM <= FIN_SMEM, "a direct run's record sort fits the staged records' limit");

template <int LK, int D>
int launch_d(FinArgs &a, cudaStream_t st) {
  auto kern = k_finish<LK, D>;
  // capacity of the staged lists and the shared memory they take
  a.Kc = (a.K + 31) & ~31;
  size_t smem = (size_t)a.Kc * fin_record_bytes(D);
  if (a.out) {  // the record sort reuses it
    smem = std::max(smem, (size_t)fin_pow2(a.n_rec) * REC_BYTES);
  }
  // blocks: a search is K / 32 steps of one warp, so few clusters need few blocks, and
  // the lines leave the other SMs free where more bring nothing (whole runs, ms, with
  // 1 / 4 / 8 / 16 blocks: 2-D Ward 96 clusters 0.192 / 0.188 / 0.188 / 0.189, 320 0.286 /
  // 0.261 / 0.262 / 0.254, 640 0.434 / 0.335 / 0.322 / 0.312, 2,000 1.52 / 0.73 / 0.59 /
  // 0.53; 16-D 2,000 5.2 / 2.2 / 1.8 / 1.5)
  const int nct = a.K <= 96 ? 1 : a.K <= 320 ? 4 : a.K <= 640 ? 8 : 16;
  return launch_cluster((const void *)kern, nct, FT, smem, &a, st);
}

template <int LK>
int launch_lk_fin(FinArgs &a, cudaStream_t st) {
  switch (fin_dim(a.s.d)) {
    case 1: return launch_d<LK, 1>(a, st);
    case 2: return launch_d<LK, 2>(a, st);
    case 3: return launch_d<LK, 3>(a, st);
    case 4: return launch_d<LK, 4>(a, st);
    case 5: return launch_d<LK, 5>(a, st);
    case 6: return launch_d<LK, 6>(a, st);
    case 8: return launch_d<LK, 8>(a, st);
    case 10: return launch_d<LK, 10>(a, st);
    case 12: return launch_d<LK, 12>(a, st);
    default: return launch_d<LK, 16>(a, st);
  }
}

}  // namespace

int launch_cluster(const void *kern, int nct, int threads, size_t smem, void *args,
                   cudaStream_t st) {
  // The limit belongs to the kernel, not to this call: always the same value, so that a
  // launch of another thread is never left above it
  if (smem > 48 * 1024)
    CK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, FIN_SMEM));
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (nct > 8) CK(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  for (;; nct >>= 1) {  // 16 blocks where the device can place them, else the portable 8
    cfg.gridDim = dim3(nct);
    at.val.clusterDim.x = nct;
    if (nct <= 8) break;
    int can = 0;
    if (cudaOccupancyMaxActiveClusters(&can, kern, &cfg) == cudaSuccess && can >= 1) break;
    cudaGetLastError();
  }
  void *pa[1] = {args};
  CK(cudaLaunchKernelExC(&cfg, kern, pa));
  return HAC_OK;
}

int launch_rec_sort(const State &s, int m, hac_merge *out, int32_t *out_round, cudaStream_t st) {
  const size_t smem = (size_t)fin_pow2(m) * REC_BYTES;
  if (smem > 48 * 1024)  // (one value for every call, as in launch_cluster)
    CK(cudaFuncSetAttribute(k_rec_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, FIN_REC_SMEM));
  k_rec_sort<<<1, FT, smem, st>>>(s, m, out, out_round);
  CK(cudaGetLastError());
  return HAC_OK;
}

int launch_finish(FinArgs &a, cudaStream_t st) {
  return a.s.linkage == LK_WARD ? launch_lk_fin<LK_WARD>(a, st) : launch_lk_fin<LK_AVG2>(a, st);
}

}  // namespace hacg
