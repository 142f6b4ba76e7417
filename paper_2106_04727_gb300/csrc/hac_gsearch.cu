// Nearest-neighbour search of Ward and avg-2 for groups of terminals at once, and
// of complete and average linkage in the first round, whose pairs of single
// points are plain distances.
//
// The search of hac_query.cuh gives every terminal a warp, whose lanes share
// the tree nodes and bucket records; at 10^6 points in 5-D a search is some 25
// dependent steps of about 120 instructions, and its FP64 keys (two lanes per
// clock and SM) are computed for one terminal at a time.  Consecutive terminals
// lie next to each other in the spatial order and visit nearly the same
// buckets, so here a warp searches for G of them together: one lane per
// terminal (32 / G lanes share a terminal's records when G < 32).  Records are
// read by uniform loads, tested against every lane's own threshold in FP32, and
// a node is opened, or a bucket scanned, if any lane itself reaches its box;
// before that, all children of a node at once are pruned with the group's box,
// its smallest size and its largest threshold.  FP64 keys are
// computed once per terminal at the end, all lanes at a time.
//
// Bounds.  Every test is on FP32 squared distances of the same FP32 records, and
// a node's or group's box distance is computed by the same operations on
// coordinate differences no larger than any record's, so rounding is monotone
// and pruning needs no absolute slack.  Screening and the decision follow
// hac_finish.cu: with |D32 - D| <= delta + rho D a terminal whose second least
// lower bound exceeds the least upper bound has its winner; the others (near
// ties, a fraction of a percent) are left to the warp-per-terminal FP64 search.
// Same nearest neighbours, keys and ties as that search.
//
// The visits of a group are the union of its terminals' visits, so a larger group
// scans more records per terminal and fewer instructions per record.  Measured,
// Ward whole runs of 10^6 points (ms, group size from GS_WIDE terminals on):
// 2-D 17.0 / 17.2 / 17.2 (8 / 16 / 32), 5-D 45.6 / 47.4 / 54.3, 8-D 96.4 / 94.3 /
// 107.9; the warp-per-terminal search: 27.6, 59.5, 170.  (With the group's bounds
// alone for inner nodes.  Each lane's own test of the popped node, for groups that
// span a gap of the spatial order: 5-D 42.7 -> 33.0 with 8.)  10^7 2-D points have
// enough terminals for the widest: first round 9.8 ms with 8, 4.2 with 32 (43
// before).  Below that few groups
// leave warps idle: 60,000 points in 5-D 7.5 with 4, 8.2 with 8 (9.8 before).
// A terminal that reaches much farther than its group (a large cluster among
// singletons: a node's bound knows only its smallest size) is searched by the
// whole warp alone; leaving it in the group cost 11 of 57 ms in 5-D.  How much
// farther matters little: squared radius 2 / 4 / 8 / 16 times the group's mean (binary
// orders 1 to 4), 10^6 points: 5-D Ward 32.1 / 31.1 / 31.0 / 31.1, 2-D avg-2 11.6 /
// 10.7 / 10.3 / 10.1.
//
// A node's nearest child is visited first.  In index order a terminal alone in its
// bucket beside a dense line of points came in from the far end of the tree: whole
// Ward run of 10^7 clipped 2-D Gaussians 396 ms, 62 nearest first (202 with the
// warp-per-terminal search); 10^7 2-D spreaders 77 and 54.
#include "hac_query.cuh"

namespace hacg {

namespace {

// group sizes (from GS_WIDE terminals on in d <= 2, above, and below), how many binary orders of
// magnitude over its group's mean a squared radius may be, warps per block
#ifndef HAC_GS_W
#define HAC_GS_W 8
#endif
#ifndef HAC_GS_W2
#define HAC_GS_W2 32
#endif
#ifndef HAC_GS_N
#define HAC_GS_N 4
#endif
#ifndef HAC_GS_GW
#define HAC_GS_GW 4
#endif
#ifndef HAC_GS_CUT
#define HAC_GS_CUT 2
#endif
constexpr int GS_W2 = HAC_GS_W2, GS_W = HAC_GS_W, GS_N = HAC_GS_N;
constexpr int GW = HAC_GS_GW;         // warps per block
// entries of a depth-first stack: 32 of the top level and 31 more for each of the
// MAXLEV - 1 levels below it, 311
constexpr int GSTK = 320;

__device__ __forceinline__ float g_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// order-preserving bits of a float
__device__ __forceinline__ unsigned f_ord(float x) {
  const unsigned u = __float_as_uint(x);
  return u >> 31 ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float f_unord(unsigned o) {
  return __uint_as_float(o >> 31 ? o ^ 0x80000000u : ~o);
}

template <int D, int DP>
__device__ __forceinline__ void g_load(const float *row, float (&v)[D]) {
  if (DP == 2) {
    const float2 a = *(const float2 *)row;
    v[0] = a.x;
    if (D > 1) v[1 % D] = a.y;
  } else {
    const float4 a = *(const float4 *)row;
    v[0] = a.x;
    v[1 % D] = a.y;
    v[2 % D] = a.z;
    if (D > 3) v[3 % D] = a.w;
    if (D > 5) {
      const float4 b = *(const float4 *)(row + 4);
      v[4 % D] = b.x;
      v[5 % D] = b.y;
      if (D > 6) v[6 % D] = b.z;
      if (D > 7) v[7 % D] = b.w;
    } else if (D > 4) {
      v[4 % D] = row[4];
    }
  }
}

// One lane's terminal.  Squared-key domain: Ward w ||.||^2, avg-2 ||.||^2 + var
// + var; `g` is 1 / size (Ward) or the variance (avg-2).
template <int LK, int D>
struct GTerm {
  float x[D], g, delta, sq2n;  // sq2n: sqrt(2 |C|), the largest sqrt(w) (Ward)
  float L1, L2, U, tq;         // bounds so far, and the squared test threshold
  int p1, pos;

  // candidates whose lower bound can be within U pass dc2 <= tq (...)
  __device__ void threshold(float rho2) {
    const float r = sqrtf(U * (1.f + 2.2f * rho2)) + (LK == LK_WARD ? delta * sq2n : delta);
    tq = r * r * (1.f + 1e-5f);
  }
  // squared distance that passes beside a record (or node) with 1 / size gb
  // (largest under the node), Ward; avg-2: minus the variances
  __device__ float limit(float gb) const {
    // (single points of complete and average linkage: variances of 0)
    return LK == LK_WARD ? 0.5f * tq * (g + gb) : tq - g - gb;
  }
};

struct GCount {
  unsigned tests, nodes, offers;
};

// The search of a warp: lane l searches for terminal cid ci (one of G, repeated
// every G lanes; `act`: a real one).  Returns the lanes (below G) whose
// terminals reach so far that they are to be searched alone.
template <int LK, int D, int DP, int G>
__device__ __forceinline__ unsigned g_search(const QueryArgs &a, const int *s_ti, uint32_t *sn,
                                             float *sd, int lane, int ci, bool act, bool f32,
                                             GCount &n) {
  constexpr int S = 32 / G;  // lanes per terminal
  constexpr int B = G == 1 ? 1 : D <= 3 ? 4 : 2;
  const int slice = lane / G;
  const float rho2 = 2.2f * ((float)a.d + 16.f) * U32;
  GTerm<LK, D> T;
  T.pos = a.pos[ci];
  g_load<D, DP>(a.q32 + (size_t)T.pos * DP, T.x);
  const float fna = (float)a.qsz[T.pos];
  T.g = a.qvar[T.pos];
  T.sq2n = sqrtf(2.f * fna);
  T.delta = 2.01f * U32 * a.coord_scale * sqrtf((float)a.d) * 1.01f;
  T.L1 = T.L2 = INFINITY;
  T.p1 = -1;
  const unsigned long long pv = a.pred[ci];
  T.U = pv == PRED_EMPTY ? INFINITY : __uint_as_float((unsigned)(pv >> 32));
  T.threshold(rho2);
  const int own = a.pbkt[T.pos];
  // the group's box, largest 1 / size (Ward) or least variance (avg-2), and
  // largest threshold (bits of non-negative floats order like their values)
  float glo[D], ghi[D];
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const unsigned o = f_ord(T.x[k]);
    glo[k] = f_unord(__reduce_min_sync(0xffffffffu, o));
    ghi[k] = f_unord(__reduce_max_sync(0xffffffffu, o));
  }
  const float gg = LK == LK_WARD
                       ? __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(T.g)))
                       : __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(T.g)));
  float TQ = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(T.tq)));

  bool alone = false;
  auto scan = [&](int j) {
    const int b = a.nch[a.chb[0] + j], e = min(a.nch[a.chb[0] + j + 1], a.K);
    n.tests += (unsigned)(e - b) * G;
    bool better = false;
    // B records' loads are issued together
    for (int p0 = b + slice; p0 - slice < e; p0 += S * B) {
      float y[B][D], gb[B];
#pragma unroll
      for (int r = 0; r < B; ++r) {
        const int p = min(p0 + r * S, e - 1);
        g_load<D, DP>(a.q32 + (size_t)p * DP, y[r]);
        gb[r] = a.qvar[p];
      }
#pragma unroll
      for (int r = 0; r < B; ++r) {
        const int p = p0 + r * S;
        float dc2 = 0.f;
#pragma unroll
        for (int k = 0; k < D; ++k) {
          const float u = T.x[k] - y[r][k];
          dc2 = fmaf(u, u, dc2);
        }
        if (p >= e || p == T.pos || alone || !(dc2 <= T.limit(gb[r]))) continue;
        ++n.offers;
        float lo, up;
        if (LK == LK_WARD) {
          const float w = 2.f * g_rcp(T.g + gb[r]), q = sqrt_approx_ftz(dc2);
          const float l = fmaxf(q - T.delta, 0.f), h = q + T.delta;
          lo = w * l * l;
          up = w * h * h;
        } else {
          const float q = sqrt_approx_ftz(dc2 + T.g + gb[r]);
          const float l = fmaxf(q - T.delta, 0.f), h = q + T.delta;
          lo = l * l;
          up = h * h;
        }
        if (lo < T.L1) {
          T.L2 = T.L1;
          T.L1 = lo;
          T.p1 = p;
        } else {
          T.L2 = fminf(T.L2, lo);
        }
        if (up < T.U) {
          T.U = up;
          better = true;
        }
      }
    }
    if (__any_sync(0xffffffffu, better)) {
      if (S > 1) {  // lanes of one terminal share its U
#pragma unroll
        for (int o = G; o < 32; o <<= 1) T.U = fminf(T.U, __shfl_xor_sync(0xffffffffu, T.U, o));
      }
      if (!alone) T.threshold(rho2);
      TQ = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(T.tq)));
    }
  };

  // the terminals' own buckets first: they usually settle tight bounds
  for (unsigned left = 0xffffffffu; left;) {
    const int j = __shfl_sync(0xffffffffu, own, __ffs(left) - 1);
    left &= ~__ballot_sync(0xffffffffu, own == j);
    scan(j);
  }
  // a terminal that reaches much farther than the others would make the whole
  // group visit its nodes: it goes to a warp of its own
  if (G > 1) {
    // exponent of the squared radius beside the smallest clusters
    const float r2 = LK == LK_WARD ? 0.5f * T.tq * (T.g + 1.f) : T.tq - T.g;
    const int ex = (int)(__float_as_uint(fmaxf(r2, 0.f)) >> 23);
    const int sum = __reduce_add_sync(0xffffffffu, ex);
    alone = ex * 32 > sum + 32 * HAC_GS_CUT;
    if (alone) T.tq = 0.f;
    TQ = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(T.tq)));
  }
  // the least threshold a node needs to pass for some terminal of the group
  auto push = [&](int top, int L, int c0, int cnt) {
    const int child = c0 + lane;
    const bool in = lane < cnt && child < s_ti[L];
    float need = INFINITY;
    if (in) {
      const int node = a.lvl_base[L] + child;
      float lo[D], hi[D];
      g_load<D, DP>(a.nclo + (size_t)node * DP, lo);
      g_load<D, DP>(a.nchi + (size_t)node * DP, hi);
      float dc2 = 0.f;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        const float u = fmaxf(fmaxf(lo[k] - ghi[k], glo[k] - hi[k]), 0.f);
        dc2 = fmaf(u, u, dc2);
      }
      need = LK == LK_WARD ? 2.f * dc2 * g_rcp(gg + g_rcp((float)a.nnmin[node])) * (1.f - 1e-6f)
                           : dc2 + gg;
    }
    n.nodes += __popc(__ballot_sync(0xffffffffu, in));
    const bool ok = in && need <= TQ;
    const unsigned m = __ballot_sync(0xffffffffu, ok);
    if (top + __popc(m) > GSTK) {  // cannot happen for the level counts of tree_caps
      if (lane == 0) atomicOr(&a.ctr->err, ERR_STACK);
      return top;
    }
    // The nearest child goes on top: a terminal alone in its bucket starts without
    // a bound, and has one after the first bucket of this descent (in index order
    // it would come in from the far end of the tree, bucket by bucket).
    const unsigned kn = ok ? __float_as_uint(need) : 0xffffffffu;  // need >= 0
    const unsigned best = __reduce_min_sync(0xffffffffu, kn);
    const int fl = __ffs(__ballot_sync(0xffffffffu, ok && kn == best)) - 1;
    if (ok) {
      const int at = top + (lane == fl ? __popc(m) - 1
                                       : __popc(m & ((1u << lane) - 1u)) - (fl < lane));
      sn[at] = ((uint32_t)L << 28) | (uint32_t)child;
      sd[at] = need;
    }
    __syncwarp();
    return top + __popc(m);
  };
  const int tl = s_ti[TI_TOP] - 1;
  int top = push(0, tl, 0, min(s_ti[tl], FAN));
  while (top > 0) {
    --top;
    const uint32_t e = sn[top];
    const float need = sd[top];
    __syncwarp();
    if (need > TQ) continue;
    const int L = (int)(e >> 28), j = (int)(e & ((1u << 28) - 1));
    if (L == 0 && __any_sync(0xffffffffu, own == j)) continue;  // scanned first
    // does any terminal itself reach the node's box?  (The group's box may span
    // a gap of the spatial order, with a dense region inside it that no terminal
    // reaches.)
    const int node = a.lvl_base[L] + j;
    float lo[D], hi[D];
    g_load<D, DP>(a.nclo + (size_t)node * DP, lo);
    g_load<D, DP>(a.nchi + (size_t)node * DP, hi);
    float dc2 = 0.f;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const float u = fmaxf(fmaxf(lo[k] - T.x[k], T.x[k] - hi[k]), 0.f);
      dc2 = fmaf(u, u, dc2);
    }
    const float gb = LK == LK_WARD ? g_rcp((float)a.nnmin[node]) * (1.f + 1e-6f) : 0.f;
    if (!__any_sync(0xffffffffu, !alone && dc2 <= T.limit(gb))) continue;
    if (L > 0) {
      const int c0 = a.nch[a.chb[L] + j];
      top = push(top, L - 1, c0, a.nch[a.chb[L] + j + 1] - c0);
    } else {
      scan(j);
    }
  }
  // the lanes of one terminal together
  if (S > 1) {
#pragma unroll
    for (int o = G; o < 32; o <<= 1) {
      const float l1 = __shfl_xor_sync(0xffffffffu, T.L1, o);
      const float l2 = __shfl_xor_sync(0xffffffffu, T.L2, o);
      const int q1 = __shfl_xor_sync(0xffffffffu, T.p1, o);
      if (l1 < T.L1) {
        T.L2 = fminf(T.L1, l2);
        T.L1 = l1;
        T.p1 = q1;
      } else {
        T.L2 = fminf(T.L2, l1);
      }
    }
  }
  const float lim = T.U * (1.f + rho2);
  const bool one = T.p1 >= 0 && T.L1 * (1.f - rho2) <= lim && T.L2 * (1.f - rho2) > lim;
  if (act && slice == 0) {
    if (one && !alone) {
      const int cb = a.order[T.p1];
      double key;
      if (LK == LK_COMPLETE || LK == LK_AVERAGE) {
        // as the search of hac_query.cuh: in the FP32 mode the upper bound of the
        // FP32 distance where that is within 4e-6, else the FP64 distance
        const float d1 = f32 ? eval32_lane<LK, DP>(a.p32, a.qseg[T.pos], 1, a.qseg[T.p1], 1) : 0.f;
        const float rho = ((float)a.d + 16.f) * U32 + (LK == LK_AVERAGE ? 32.f * U32 : 0.f);
        const float e1 = a.delta_pts;
        if (f32 && e1 + rho * d1 <= 4e-6f * d1)
          key = (double)((d1 + e1) * (1.f + rho));
        else
          key = eval64_lane<LK, DP>(a.p64, a.qseg[T.pos], 1, a.qseg[T.p1], 1);
      } else {
        const int na = a.qsz[T.pos], nb = a.qsz[T.p1];
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < D; ++k) {
          if (k < a.d) {
            const double u = a.q64[(size_t)T.pos * DP + k] - a.q64[(size_t)T.p1 * DP + k];
            s += u * u;
          }
        }
        key = LK == LK_AVG2 ? s + a.sse[ci] / (double)na + a.sse[cb] / (double)nb
                            : (2.0 * (double)na * (double)nb) / (double)(na + nb) * s;
      }
      a.Ekey[ci] = key;
      a.Ecid[ci] = cb;
    } else if (!alone) {
      a.pend_out[atomicAdd(&a.ctr->nrq, 1)] = ci;
    }
  }
  __syncwarp();
  return __ballot_sync(0xffffffffu, alone && act && slice == 0);
}

template <int LK, int D, int DP, int G>
__global__ void __launch_bounds__(GW * 32) k_gsearch(QueryArgs a, bool f32) {
  __shared__ uint32_t s_node[GW][GSTK];
  __shared__ float s_need[GW][GSTK];
  __shared__ int s_ti[TI_SIZE];
  for (int i = threadIdx.x; i < TI_SIZE; i += blockDim.x) s_ti[i] = a.tinfo[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int top = s_ti[TI_TOP] - 1;
  if (top < 0 || top > MAXLEV) {  // never for a finished build
    if (threadIdx.x == 0) atomicOr(&a.ctr->err, ERR_TREE);
    return;
  }
  const int t0 = (blockIdx.x * GW + wib) * G;
  if (t0 >= a.nterm) return;
  const int t = t0 + lane % G;
  const int ci = a.term[min(t, a.nterm - 1)];
  GCount n{0, 0, 0};
  unsigned far = g_search<LK, D, DP, G>(a, s_ti, s_node[wib], s_need[wib], lane, ci,
                                        t < a.nterm, f32, n);
  for (; far; far &= far - 1)
    g_search<LK, D, DP, 1>(a, s_ti, s_node[wib], s_need[wib], lane,
                           __shfl_sync(0xffffffffu, ci, __ffs(far) - 1), true, f32, n);
  n.offers = __reduce_add_sync(0xffffffffu, n.offers);
  if (lane == 0) {
    atomicAdd(&a.ctr->cluster_pairs, (unsigned long long)n.offers);
    atomicAdd(&a.ctr->nodes, (unsigned long long)n.nodes);
    atomicAdd(&a.ctr->ltests, (unsigned long long)n.tests);
  }
}

template <int LK, int D>
cudaError_t launch_g(const QueryArgs &a, bool f32, cudaStream_t s) {
  constexpr int DP = D <= 2 ? 2 : D <= 4 ? 4 : 8;
  constexpr int W = D <= 2 ? GS_W2 : GS_W;
  const bool wide = a.nterm >= GS_WIDE;
  const int G = wide ? W : GS_N;
  const int groups = (a.nterm + G - 1) / G;
  const int blocks = (groups + GW - 1) / GW;
  if (wide)
    k_gsearch<LK, D, DP, W><<<blocks, GW * 32, 0, s>>>(a, f32);
  else
    k_gsearch<LK, D, DP, GS_N><<<blocks, GW * 32, 0, s>>>(a, f32);
  return cudaGetLastError();
}

template <int LK>
cudaError_t launch_glk(const QueryArgs &a, bool f32, cudaStream_t s) {
  switch (a.d) {
    case 1: return launch_g<LK, 1>(a, f32, s);
    case 2: return launch_g<LK, 2>(a, f32, s);
    case 3: return launch_g<LK, 3>(a, f32, s);
    case 4: return launch_g<LK, 4>(a, f32, s);
    case 5: return launch_g<LK, 5>(a, f32, s);
    case 6: return launch_g<LK, 6>(a, f32, s);
    case 7: return launch_g<LK, 7>(a, f32, s);
    case 8: return launch_g<LK, 8>(a, f32, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_gsearch(const QueryArgs &a, int prec, cudaStream_t s) {
  if (a.nterm <= 0) return cudaSuccess;
  const bool f32 = prec != 0;
  switch (a.linkage) {
    case LK_COMPLETE: return launch_glk<LK_COMPLETE>(a, f32, s);
    case LK_AVERAGE: return launch_glk<LK_AVERAGE>(a, f32, s);
    case LK_WARD: return launch_glk<LK_WARD>(a, f32, s);
    case LK_AVG2: return launch_glk<LK_AVG2>(a, f32, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hacg
