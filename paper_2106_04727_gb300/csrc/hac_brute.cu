// Exhaustive nearest-neighbour search for the closed-form linkages (Ward,
// avg-2) in high dimension.
//
// In d > 8 the spatial tree of hac_query.cuh prunes little (most node boxes
// overlap every query ball), so every terminal looks at every active cluster.
// What a pair must pay is one contraction over the coordinates: the tensor
// cores take it (k_gram), and only pairs that may matter are scored in FP32.
//
//   k_gram_seed  U = least upper bound among the predecessor bound and 32
//                neighbours in the spatial order;
//   k_gram       blocks of 256 terminals stream all records.  Rows and columns
//                are recentred on the block's own box, scaled to FP16, and
//                x . y comes from m16n8k16 tensor instructions with FP32
//                accumulation.  With nx, ny the FP32 squared norms,
//                  ||x - y||^2 >= (nx + ny)(1 - eps) - 2 x . y,
//                eps = 1.03 * 2^-10: each FP16 rounding is within 2^-11 of its
//                coordinate, so the product sum is within (2^-10 + 2^-22)
//                ||x|| ||y|| <= (2^-11 + 2^-23)(nx + ny), and the FP32
//                accumulation within 2^-18 of that.  (A scaled coordinate below
//                2^-14 is a subnormal FP16 number, off by up to 2^-25 and not by
//                2^-11 of itself: against a coordinate above 2^-9 the spare 0.03 of
//                eps covers that, else the delta added to the threshold's root, at
//                least 2^-12 sqrt(d) here.)  A pair whose bound is
//                within the terminal's threshold is scored in FP32 exactly as
//                the search does (|D32 - D| <= delta + rho D) and, if its lower
//                bound is within U, goes on the terminal's list;
//   k_gram_fin   the candidates listed within the final U: one wins outright,
//                more are compared by their FP64 keys, least (key, cid).  A
//                list that overflowed is left to k_brute_recheck, a tiled pass
//                that re-scores in FP64 every candidate within U.
//
// The result is the same (key, cid) the tree search returns.  Single
// instance only (all active clusters are candidates).
//
// Bound by the tensor instructions (4 per 64 x 8 pairs) and the 1 to 1.5
// comparisons a pair still costs.  The scalar scan this replaces (32 FP32
// operations a pair) took 53.9 ms for the first round of 150,000 16-D points,
// this 4.4; the whole avg-2 run 270 ms, now 25.7.
#include "hac_query.cuh"

#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

namespace hacg {

namespace {

// tile shape (the tuner's compiled variants override these)
#ifndef HAC_BR_T
#define HAC_BR_T 256
#endif
#ifndef HAC_BR_C
#define HAC_BR_C 128
#endif
constexpr int BR_T = HAC_BR_T;  // terminals per CTA
constexpr int BR_C = HAC_BR_C;  // candidate records per staged tile

template <int LK, int DP>
struct BruteTerm {
  int ci, na, mypos;
  float fna, vA, delta0, rho;
  float x[DP];

  __device__ void init(const QueryArgs &a, int c) {
    ci = c;
    na = a.csize[ci];
    fna = (float)na;
    mypos = a.pos[ci];
    vA = LK == LK_AVG2 ? a.qvar[mypos] : 0.f;
#pragma unroll
    for (int k = 0; k < DP; ++k) x[k] = a.cent32[(size_t)ci * DP + k];
    delta0 = 2.01f * U32 * a.iscale[a.inst[ci]] * sqrtf((float)a.d);
    rho = ((float)a.d + 16.f) * U32;
  }

  // FP32 distance (D units) of the candidate staged at q with size / variance
  // sv, and its absolute error term
  __device__ void score(const float *q, float sv, float &d32, float &dlt) const {
    float dc2 = 0.f;
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const float t = x[k] - q[k];
      dc2 = fmaf(t, t, dc2);
    }
    if (LK == LK_WARD) {
      const float w = ward_w(fna, sv);
      d32 = sqrtf(w * dc2);
      dlt = delta0 * sqrtf(w);
    } else {
      d32 = sqrtf(dc2 + vA + sv);
      dlt = delta0;
    }
  }

  __device__ float lower(float d32, float dlt) const { return fmaxf(d32 - dlt, 0.f) * (1.f - rho); }

  // Cheap test that a candidate's lower bound exceeds u, with no root or
  // division: lo <= u needs D32 <= u / (1 - rho) + dlt, and dlt is at most
  // dmax (Ward: delta0 sqrt(w) with w <= 2|C_i|), so a candidate whose
  // squared FP32 distance exceeds tau = (u / (1 - rho) + dmax)^2 (widened by
  // 1e-5 for the rounding of this test) cannot pass.  Ward compares
  // 2|A||B| dc2 > tau (|A| + |B|) to avoid the division in w.
  __device__ float tau(float u) const {
    if (!(u < INFINITY)) return INFINITY;
    const float dmax = LK == LK_WARD ? delta0 * sqrtf(2.f * fna) : delta0;
    const float r = u / (1.f - rho) + dmax;
    return r * r * (1.f + 1e-5f);
  }

  __device__ bool beyond(const float *q, float sv, float tq) const {
    float dc2 = 0.f;
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      const float t = x[k] - q[k];
      dc2 = fmaf(t, t, dc2);
    }
    if (LK == LK_WARD) return 2.f * fna * sv * dc2 > tq * (fna + sv);
    return dc2 + vA + sv > tq;
  }

  // FP64 key of candidate cb (by cid), as the tree search computes it
  __device__ unsigned long long exact(const QueryArgs &a, int cb) const {
    double cA[DP], cB[DP];
#pragma unroll
    for (int k = 0; k < DP; ++k) {
      cA[k] = a.cent[(size_t)ci * DP + k];
      cB[k] = a.cent[(size_t)cb * DP + k];
    }
    const int nb = a.csize[cb];
    if (LK == LK_AVG2) {
      double g2 = 0.0;
#pragma unroll
      for (int k = 0; k < DP; ++k) {
        const double t = cA[k] - cB[k];
        g2 += t * t;
      }
      return kbits(g2 + a.sse[ci] / (double)na + a.sse[cb] / (double)nb);
    }
    return kbits(ward_key<DP>(cA, cB, na, nb, DP));
  }
};

// Stage candidate records [p0, p0 + BR_C) of the active order.
template <int LK, int DP>
__device__ __forceinline__ int stage(const QueryArgs &a, int p0, float *sq, float *sv, int *sc) {
  const int cnt = min(BR_C, a.K - p0);
  for (int i = threadIdx.x; i < cnt * DP; i += BR_T) sq[i] = a.q32[(size_t)p0 * DP + i];
  for (int j = threadIdx.x; j < cnt; j += BR_T) {
    sc[j] = a.order[p0 + j];
    sv[j] = LK == LK_WARD ? (float)a.qsz[p0 + j] : a.qvar[p0 + j];
  }
  return cnt;
}

// ---------------------------------------------------------------------------
// tensor-core screening
// ---------------------------------------------------------------------------
constexpr int GR = 256;       // terminals (rows) per block
constexpr int GC = 128;       // records (columns) per staged tile
constexpr int GT = 256;       // threads: 8 warps, warp w has rows 64 (w % 4) and
                              // half w / 4 of the tile's columns
constexpr int GQ = 64 * 16;   // survivors of one warp step (64 rows x 16 columns)
constexpr float G_EPS = 1.03f / 1024.f;

struct GramArgs {
  float scl;    // coordinates times 2^k lie within 2^13
  int tiles;    // tiles of GC records per split
};

__device__ __forceinline__ void mma_f16(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                        unsigned b1, float c0, float c1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%11,%10,%11};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c0), "f"(c1));
}

__device__ __forceinline__ void ldsm4(unsigned (&r)[4], const void *p) {
  const unsigned at = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(at));
}

// eight coordinates, recentred and scaled: their FP16 pairs and squared norm
__device__ __forceinline__ float gram_pack(const float (&v)[8], const float *ctr, float scl,
                                           uint4 &out) {
  float n = 0.f;
  unsigned w[4];
#pragma unroll
  for (int k = 0; k < 8; k += 2) {
    const float x = (v[k] - ctr[k]) * scl, y = (v[k + 1] - ctr[k + 1]) * scl;
    n = fmaf(x, x, fmaf(y, y, n));
    const __half2 h = __floats2half2_rn(x, y);
    w[k / 2] = *(const unsigned *)&h;
  }
  out = make_uint4(w[0], w[1], w[2], w[3]);
  return n;
}

template <int DP>
__device__ __forceinline__ void gram_load(const float *row, int half, bool in, float (&v)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = 0.f;
  if (in && half * 8 < DP) {
    const float4 a = *(const float4 *)(row + half * 8), b = *(const float4 *)(row + half * 8 + 4);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  }
}

// U of every terminal from its predecessor and 32 neighbours in the order
template <int LK, int DP>
__global__ void k_gram_seed(QueryArgs a) {
  const int lane = threadIdx.x & 31;
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (t >= a.nterm) return;
  BruteTerm<LK, DP> T;
  T.init(a, a.term[t]);
  const int q = T.mypos - 16 + lane + (lane >= 16);
  float up = INFINITY;
  if (q >= 0 && q < a.K) {
    float d32, dlt;
    T.score(a.q32 + (size_t)q * DP, LK == LK_WARD ? (float)a.qsz[q] : a.qvar[q], d32, dlt);
    up = (d32 + dlt) * (1.f + T.rho);
  }
  up = warp_minf(up);
  if (lane == 0) {
    const unsigned long long pv = a.pred[T.ci];
    if (pv != PRED_EMPTY)
      up = fminf(up, __fsqrt_ru(__uint_as_float((unsigned)(pv >> 32))));
    a.gu[t] = up;
    a.gcnt[t] = 0;
  }
}

// One block: its 256 terminals against the records of split blockIdx.y.
template <int LK, int DP>
__global__ void __launch_bounds__(GT, 2) k_gram(QueryArgs a, GramArgs g) {
  __shared__ __align__(16) unsigned char s_b[2][2][GC * 16];  // [buffer][k half][column][8]
  __shared__ __align__(8) float s_h[2][GC];   // -(ny (1 - eps) + scaled variance) / 2
  __shared__ __align__(8) float s_g[2][GC];   // Ward: 1 / size
  __shared__ float s_x[GR][DP + 1];           // the terminals' FP32 centroids
  __shared__ float s_nx[GR], s_ga[GR], s_dm[GR], s_thr[GR], s_kq[GR];
  __shared__ unsigned s_u[GR];                // U (bits of a non-negative float)
  __shared__ int s_pos[GR];
  __shared__ unsigned short s_q[GT / 32][GQ];
  __shared__ int s_qn[GT / 32];
  __shared__ unsigned s_lo[DP], s_hi[DP];
  __shared__ float s_c[16];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int t0 = blockIdx.x * GR, t = t0 + tid;
  const bool act = t < a.nterm;
  const int ins = a.inst[a.term[t0]];
  const float delta0 = 2.01f * U32 * a.iscale[ins] * sqrtf((float)a.d);
  const float rho = ((float)a.d + 16.f) * U32;
  // rows: FP32 records, box centre, FP16 fragments
  if (tid < DP) {
    s_lo[tid] = ~0u;
    s_hi[tid] = 0u;
  }
  __syncthreads();
  const int ci = act ? a.term[t] : a.term[t0];
  const int mp = a.pos[ci];
  const float fna = (float)a.csize[ci];
#pragma unroll
  for (int k = 0; k < DP; ++k) {
    const float x = a.cent32[(size_t)ci * DP + k];
    s_x[tid][k] = x;
    const unsigned u = __float_as_uint(x), o = u >> 31 ? ~u : u | 0x80000000u;  // order-preserving
    const unsigned mn = __reduce_min_sync(0xffffffffu, o), mx = __reduce_max_sync(0xffffffffu, o);
    if (lane == 0) {
      atomicMin(&s_lo[k], mn);
      atomicMax(&s_hi[k], mx);
    }
  }
  __syncthreads();
  if (tid < 16) {
    float c = 0.f;
    if (tid < DP) {
      const unsigned l = s_lo[tid], h = s_hi[tid];
      c = 0.5f * (__uint_as_float(l >> 31 ? l ^ 0x80000000u : ~l) +
                  __uint_as_float(h >> 31 ? h ^ 0x80000000u : ~h));
    }
    s_c[tid] = c;
  }
  __syncthreads();
  unsigned af[4][4];
  {
    // rows through the column buffers, 64 rows of one warp pair at a time
    const float s2 = g.scl * g.scl;
    float nx = 0.f;
    uint4 hv[2];
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = hf * 8 + k < DP ? s_x[tid][hf * 8 + k < DP ? hf * 8 + k : 0] : 0.f;
      nx += gram_pack(v, s_c + hf * 8, g.scl, hv[hf]);
    }
    // (a row past the last terminal passes nothing)
    s_nx[tid] = !act ? INFINITY : 0.5f * (nx * (1.f - G_EPS) + (LK == LK_AVG2 ? a.qvar[mp] * s2 : 0.f));
    s_ga[tid] = 1.f / fna;
    s_dm[tid] = 2.f * (LK == LK_WARD ? delta0 * sqrtf(2.f * fna) : delta0);
    s_u[tid] = act ? __float_as_uint(a.gu[t]) : 0u;
    s_pos[tid] = mp;
    // 256 rows x 2 halves of 16 B: rows [0, 128) in buffer 0, [128, 256) in buffer 1
    *(uint4 *)&s_b[tid >> 7][0][(tid & 127) * 16] = hv[0];
    *(uint4 *)&s_b[tid >> 7][1][(tid & 127) * 16] = hv[1];
    __syncthreads();
    const int r0 = (w & 3) * 64;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      // matrices: rows 0-7 k 0-7, rows 8-15 k 0-7, rows 0-7 k 8-15, rows 8-15 k 8-15
      const int row = r0 + m * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
      ldsm4(af[m], &s_b[row >> 7][lane >> 4][(row & 127) * 16]);
    }
  }
  // thresholds of this warp's 64 rows from U: see the header of this file;
  // the recentring rounds once more, hence twice delta
  auto thresholds = [&]() {
#pragma unroll
    for (int r = lane; r < 64; r += 32) {
      const int row = (w & 3) * 64 + r;
      const float u = __uint_as_float(*(volatile unsigned *)&s_u[row]);
      const float rr = u / (1.f - rho) + s_dm[row];
      const float tau = rr * rr * (1.f + 1e-5f) * g.scl * g.scl;  // may be inf: all pass
      if (LK == LK_WARD) {
        s_kq[row] = 0.25f * tau;
        s_thr[row] = s_nx[row] - 0.25f * tau * s_ga[row];
      } else {
        s_thr[row] = s_nx[row] - 0.5f * tau;
      }
    }
    __syncwarp();
  };
  float thr[8], kq[8];
  auto reload = [&]() {
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = (w & 3) * 64 + m * 16 + h * 8 + (lane >> 2);
        thr[m * 2 + h] = s_thr[row];
        kq[m * 2 + h] = LK == LK_WARD ? s_kq[row] : 0.f;
      }
  };
  thresholds();
  reload();
  if (lane == 0) s_qn[w] = 0;
  __syncthreads();  // the row fragments are read: the buffers are free

  const int nt = (a.K + GC - 1) / GC;
  const int tile0 = blockIdx.y * g.tiles, tile1 = min(nt, tile0 + g.tiles);
  // the block's own region of the order first, where it lies in this split
  const int own = s_pos[0] / GC;
  const int start = own >= tile0 && own < tile1 ? own : tile0;
  const int cnt = tile1 - tile0;
  auto tile_at = [&](int it) {
    const int x = start + it;
    return x < tile1 ? x : x - cnt;
  };
  const int col = tid >> 1, half = tid & 1;
  float nv[8], nsv = 0.f;
  auto fetch = [&](int tl) {
    const int p = tl * GC + col;
    gram_load<DP>(a.q32 + (size_t)p * DP, half, p < a.K, nv);
    if (half == 0) nsv = p < a.K ? (LK == LK_WARD ? (float)a.qsz[p] : a.qvar[p]) : 1.f;
  };
  auto put = [&](int tl, int buf) {
    uint4 hv;
    float n = gram_pack(nv, s_c + half * 8, g.scl, hv);
    n += __shfl_xor_sync(0xffffffffu, n, 1);
    *(uint4 *)&s_b[buf][half][col * 16] = hv;
    if (half == 0) {
      const bool in = tl * GC + col < a.K;
      const float x = n * (1.f - G_EPS) + (LK == LK_AVG2 ? nsv * g.scl * g.scl : 0.f);
      s_h[buf][col] = in ? -0.5f * x : -INFINITY;
      if (LK == LK_WARD) s_g[buf][col] = 1.f / nsv;
    }
  };
  unsigned scored = 0;
  if (cnt > 0) {
    fetch(tile_at(0));
    put(tile_at(0), 0);
  }
  __syncthreads();
  for (int it = 0; it < cnt; ++it) {
    const int buf = it & 1, tl = tile_at(it);
    if (it + 1 < cnt) fetch(tile_at(it + 1));
#pragma unroll 1
    for (int np = 0; np < 4; ++np) {  // 16 columns a step
      const int c0 = (w >> 2) * 64 + np * 16;
      unsigned bf[4];
      ldsm4(bf, &s_b[buf][(lane >> 3) & 1][(c0 + (lane >> 4) * 8 + (lane & 7)) * 16]);
      const int cc = c0 + (lane & 3) * 2;
      const float2 h0 = *(const float2 *)&s_h[buf][cc], h1 = *(const float2 *)&s_h[buf][cc + 8];
      float2 g0 = make_float2(0.f, 0.f), g1 = g0;
      if (LK == LK_WARD) {
        g0 = *(const float2 *)&s_g[buf][cc];
        g1 = *(const float2 *)&s_g[buf][cc + 8];
      }
      float v[4][8];  // fragment of columns cc, cc + 1, then of cc + 8, cc + 9
      bool any = false;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        float x[4], y[4];
        mma_f16(x, af[m], bf[0], bf[1], h0.x, h0.y);
        mma_f16(y, af[m], bf[2], bf[3], h1.x, h1.y);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          float *o = &v[m][q * 4];
          o[0] = x[q * 2], o[1] = x[q * 2 + 1], o[2] = y[q * 2], o[3] = y[q * 2 + 1];
          if (LK == LK_WARD) {
            const float kk = kq[m * 2 + q];
            o[0] = fmaf(kk, g0.x, o[0]);
            o[1] = fmaf(kk, g0.y, o[1]);
            o[2] = fmaf(kk, g1.x, o[2]);
            o[3] = fmaf(kk, g1.y, o[3]);
          }
          // one comparison per row and four columns
          any |= fmaxf(fmaxf(fmaxf(o[0], o[1]), o[2]), o[3]) >= thr[m * 2 + q];
        }
      }
      if (!__any_sync(0xffffffffu, any)) continue;
      {
        // survivors: queue them, score them one per lane
        if (any) {
#pragma unroll
          for (int m = 0; m < 4; ++m)
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if (v[m][q] >= thr[m * 2 + (q >> 2)]) {
                const int row = m * 16 + (q >> 2) * 8 + (lane >> 2);
                const int cq = cc + ((q >> 1) & 1) * 8 + (q & 1);
                s_q[w][atomicAdd(&s_qn[w], 1)] = (unsigned short)(row << 7 | cq);
              }
        }
        __syncwarp();
        const int nq = s_qn[w];
        for (int i = lane; i < nq; i += 32) {
          const int row = (w & 3) * 64 + (s_q[w][i] >> 7), p = tl * GC + (s_q[w][i] & 127);
          if (t0 + row >= a.nterm || p >= a.K || p == s_pos[row]) continue;
          ++scored;
          const float *y = a.q32 + (size_t)p * DP;
          float dc2 = 0.f;
#pragma unroll
          for (int k = 0; k < DP; ++k) {
            const float d = s_x[row][k] - y[k];
            dc2 = fmaf(d, d, dc2);
          }
          float d32, dlt;
          if (LK == LK_WARD) {
            const float ww = ward_w(1.f / s_ga[row], (float)a.qsz[p]);
            d32 = sqrtf(ww * dc2);
            dlt = delta0 * sqrtf(ww);
          } else {
            d32 = sqrtf(dc2 + a.qvar[s_pos[row]] + a.qvar[p]);
            dlt = delta0;
          }
          const float lo = fmaxf(d32 - dlt, 0.f) * (1.f - rho), up = (d32 + dlt) * (1.f + rho);
          if (lo > __uint_as_float(*(volatile unsigned *)&s_u[row])) continue;
          // the other splits' improvements come back with the atomic
          const unsigned ub = __float_as_uint(up);
          const unsigned old = atomicMin((unsigned *)&a.gu[t0 + row], ub);
          atomicMin(&s_u[row], min(old, ub));
          if (lo > __uint_as_float(old)) continue;
          const int at = atomicAdd(&a.gcnt[t0 + row], 1);
          if (at < GRAM_LIST) a.glist[(size_t)(t0 + row) * GRAM_LIST + at] = p;
        }
        __syncwarp();
        if (lane == 0) s_qn[w] = 0;
        thresholds();
        reload();
      }
    }
    if (it + 1 < cnt) put(tile_at(it + 1), buf ^ 1);
    __syncthreads();
  }
  scored = __reduce_add_sync(0xffffffffu, scored);
  if (lane == 0 && scored) atomicAdd(&a.ctr->cluster_pairs, (unsigned long long)scored);
  if (tid == 0) {
    const int c_lo = tile0 * GC, c_hi = min(a.K, tile1 * GC);
    atomicAdd(&a.ctr->ltests, (unsigned long long)min(GR, a.nterm - t0) *
                                  (unsigned long long)max(0, c_hi - c_lo));
  }
}

// The winner among the listed candidates, one thread per terminal.
template <int LK, int DP>
__global__ void k_gram_fin(QueryArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.nterm) return;
  BruteTerm<LK, DP> T;
  T.init(a, a.term[t]);
  const float U = a.gu[t];
  const int n = a.gcnt[t];
  if (n > GRAM_LIST) {  // overflowed: the FP64 pass over all candidates decides
    a.Ekey[T.ci] = (double)U;
    a.pend_out[atomicAdd(&a.ctr->npend, 1)] = T.ci;
    return;
  }
  const int32_t *L = a.glist + (size_t)t * GRAM_LIST;
  unsigned long long bk = KINF, rechecks = 0;
  int bc = INT_MAX, only = -1, win = 0;
  for (int i = 0; i < n; ++i) {
    const int p = L[i];
    float d32, dlt;
    T.score(a.q32 + (size_t)p * DP, LK == LK_WARD ? (float)a.qsz[p] : a.qvar[p], d32, dlt);
    if (T.lower(d32, dlt) > U) continue;
    if (++win == 1) {
      only = p;
      continue;
    }
    for (int e = win == 2 ? 0 : 1; e < 2; ++e) {  // the first one too, once it has company
      const int cb = a.order[e ? p : only];
      const unsigned long long k = T.exact(a, cb);
      ++rechecks;
      if (kless(k, cb, bk, bc)) {
        bk = k;
        bc = cb;
      }
    }
  }
  if (win == 1) {
    bc = a.order[only];
    bk = T.exact(a, bc);
  }
  a.Ekey[T.ci] = __longlong_as_double((long long)bk);
  a.Ecid[T.ci] = bc == INT_MAX ? -1 : bc;
  if (bc == INT_MAX) atomicOr(&a.ctr->err, ERR_NO_NN);
  if (rechecks) atomicAdd(&a.ctr->rechecks, rechecks);
}

// FP64 re-score of the listed terminals: every candidate whose FP32 lower
// bound is within U, least (FP64 key, cid) wins.
template <int LK, int DP>
__global__ void __launch_bounds__(BR_T) k_brute_recheck(QueryArgs a) {
  __shared__ float sq[BR_C * DP];
  __shared__ float sv[BR_C];
  __shared__ int sc[BR_C];
  const int m = a.ctr->npend;
  if ((int)(blockIdx.x * BR_T) >= m) return;  // uniform over the CTA
  const int t = blockIdx.x * BR_T + threadIdx.x;
  const bool act = t < m;
  BruteTerm<LK, DP> T;
  float U = 0.f, tq = 0.f;
  if (act) {
    T.init(a, a.pend_out[t]);
    U = (float)a.Ekey[T.ci];
    tq = T.tau(U);
  }
  unsigned long long bk = KINF, rechecks = 0;
  int bc = INT_MAX;
  for (int p0 = 0; p0 < a.K; p0 += BR_C) {
    __syncthreads();
    const int cnt = stage<LK, DP>(a, p0, sq, sv, sc);
    __syncthreads();
    if (!act) continue;
    for (int j = 0; j < cnt; ++j) {
      if (p0 + j == T.mypos || T.beyond(sq + j * DP, sv[j], tq)) continue;
      float d32, dlt;
      T.score(sq + j * DP, sv[j], d32, dlt);
      if (T.lower(d32, dlt) > U) continue;
      const int cb = sc[j];
      const unsigned long long k = T.exact(a, cb);
      ++rechecks;
      if (kless(k, cb, bk, bc)) {
        bk = k;
        bc = cb;
      }
    }
  }
  if (!act) return;
  a.Ekey[T.ci] = __longlong_as_double((long long)bk);
  a.Ecid[T.ci] = bc == INT_MAX ? -1 : bc;
  if (bc == INT_MAX) atomicOr(&a.ctr->err, ERR_NO_NN);
  atomicAdd(&a.ctr->rechecks, rechecks);
}

// ---------------------------------------------------------------------------
// Candidate lists for average linkage (Euclidean) in high dimension.
//
// Average linkage needs point pairs, so the exhaustive scan cannot score
// candidates itself; it replaces only the tree traversal.  Each terminal (one
// thread) streams every active cluster's FP32 record through shared memory,
// as above, and keeps:
//   U  = the least upper bound on D(C_i, B) over all B: the predecessor bound
//        beta (Algorithm 2) and the Jensen bound of each record,
//        mean ||x - y|| <= sqrt(||c_A - c_B||^2 + var A + var B), with the
//        FP32 centroid distance widened by its error bound;
//   the positions of the clusters whose centroid lower bound
//        ||c_A - c_B|| <= D(A, B) (Section 4.2) is within U (times 1 + 1e-5,
//        plus the search's absolute slack): the only clusters that can be the
//        nearest neighbour.
// The list (sorted by lower bound) and U go to the warp search, which
// evaluates those candidates as it would evaluate a tree leaf.  Tiles start at
// the CTA's own region of the spatial order, so U drops early and the list
// stays short; a list longer than BL_CAP is dropped (count -1) and that
// terminal searches the tree.
// ---------------------------------------------------------------------------
template <int DP>
__global__ void __launch_bounds__(BR_T) k_cand_avg(QueryArgs a, int32_t *lpos, float *llb,
                                                   int32_t *lcnt, float *lub) {
  constexpr int H = DP / 2;
  __shared__ __align__(16) float sq[BR_C * DP];
  __shared__ float sv[BR_C];
  const int t = blockIdx.x * BR_T + threadIdx.x;
  const bool act = t < a.nterm;
  int ci = -1, mypos = -1;
  unsigned long long x[H];
  float vA = 0.f, U = INFINITY, delta0 = 0.f, rho = 0.f, slack = 0.f;
  if (act) {
    ci = a.term[t];
    mypos = a.pos[ci];
    vA = a.qvar[mypos];
#pragma unroll
    for (int h = 0; h < H; ++h)
      x[h] = ((const unsigned long long *)(a.cent32 + (size_t)ci * DP))[h];
    const unsigned long long pv = a.pred[ci];
    if (pv != PRED_EMPTY) U = __uint_as_float((unsigned)(pv >> 32));
    const int ins = a.inst[ci];
    delta0 = 2.01f * U32 * a.iscale[ins] * sqrtf((float)a.d);
    rho = ((float)a.d + 16.f) * U32 + 32.f * U32;
    slack = a.islack[ins] * 2.f;
  }
  // candidate threshold on the squared centroid distance for the current U
  auto thr2 = [&](float u) {
    if (!(u < INFINITY)) return INFINITY;
    const float tt = u * (1.f + EPS) + slack;
    return tt * tt * (1.f + 1e-6f);
  };
  float T2 = thr2(U);
  int32_t *L = act ? lpos + (size_t)mypos * BL_CAP : nullptr;
  float *LB = act ? llb + (size_t)mypos * BL_CAP : nullptr;
  int cnt = 0;
  bool over = false;
  const int nt = (a.K + BR_C - 1) / BR_C;
  const int k0 = a.pos[a.term[blockIdx.x * BR_T]] / BR_C;  // the CTA's own region first
  unsigned long long scanned = 0;
  for (int it = 0; it < nt; ++it) {
    const int p0 = ((k0 + it) % nt) * BR_C;
    const int n_here = min(BR_C, a.K - p0);
    __syncthreads();
    for (int i = threadIdx.x; i < n_here * DP; i += BR_T) sq[i] = a.q32[(size_t)p0 * DP + i];
    for (int j = threadIdx.x; j < n_here; j += BR_T) sv[j] = a.qvar[p0 + j];
    __syncthreads();
    if (!act || over) continue;
    scanned += n_here;
    for (int j = 0; j < n_here; ++j) {
      if (p0 + j == mypos) continue;
      const unsigned long long *y = (const unsigned long long *)(sq + j * DP);
      unsigned long long tt = f2_sub(x[0], y[0]);
      unsigned long long d2 = f2_mul(tt, tt);
#pragma unroll
      for (int h = 1; h < H; ++h) {
        tt = f2_sub(x[h], y[h]);
        d2 = f2_fma(tt, tt, d2);
      }
      const float dc2 = f2_hsum(d2);
      if (dc2 <= T2) {
        if (cnt == BL_CAP) {  // full: keep only what the current U still admits
          const float tl = sqrtf(T2);
          int k = 0;
          for (int q = 0; q < cnt; ++q)
            if (LB[q] <= tl) {
              L[k] = L[q];
              LB[k] = LB[q];
              ++k;
            }
          cnt = k;
        }
        if (cnt < BL_CAP) {
          L[cnt] = p0 + j;
          LB[cnt] = sqrtf(dc2);
          ++cnt;
        } else {
          over = true;
          break;
        }
      }
      // Jensen upper bound (rounded up), only when it can lower U
      const float vB = sv[j];
      if (dc2 + vA + vB < U * U) {
        const float r = __fadd_ru(__fmul_ru(__fsqrt_ru(dc2), 1.f + rho), delta0);
        const float ub = __fsqrt_ru(__fadd_ru(__fadd_ru(__fmul_ru(r, r), vA), vB));
        if (ub < U) {
          U = ub;
          T2 = thr2(U);
        }
      }
    }
  }
  if (!act) return;
  if (!over) {
    // final filter, then insertion sort by lower bound
    const float tl = sqrtf(T2);
    int k = 0;
    for (int q = 0; q < cnt; ++q)
      if (LB[q] <= tl) {
        const int pq = L[q];
        const float lq = LB[q];
        int w = k++;
        while (w > 0 && LB[w - 1] > lq) {
          L[w] = L[w - 1];
          LB[w] = LB[w - 1];
          --w;
        }
        L[w] = pq;
        LB[w] = lq;
      }
    cnt = k;
  }
  lcnt[mypos] = over ? -1 : cnt;
  lub[mypos] = U;
  atomicAdd(&a.ctr->ltests, scanned);
}

template <int LK, int DP>
cudaError_t launch_brute_dp(const QueryArgs &a, int sms, cudaStream_t s) {
  GramArgs g{};
  // coordinates (twice the largest, after the recentring) within 2^13 of FP16's 2^16
  g.scl = ldexpf(1.f, 12 - (int)ceilf(log2f(a.coord_scale)));
  const int rows = (a.nterm + GR - 1) / GR, nt = (a.K + GC - 1) / GC;
  // the records are split over blocks too, so that even few row blocks fill the
  // SMs (two blocks each) and the last wave is short: 8 blocks per SM in all,
  // but a split of at least 16 tiles, which its prologue and its own start
  // from the seeds' U cost little beside
  const int splits = std::max(1, std::min((8 * sms + rows - 1) / rows, nt / 16));
  g.tiles = (nt + splits - 1) / splits;
  k_gram_seed<LK, DP><<<(a.nterm + 7) / 8, 256, 0, s>>>(a);
  k_gram<LK, DP><<<dim3(rows, (nt + g.tiles - 1) / g.tiles), GT, 0, s>>>(a, g);
  k_gram_fin<LK, DP><<<(a.nterm + 127) / 128, 128, 0, s>>>(a);
  k_brute_recheck<LK, DP><<<(a.nterm + BR_T - 1) / BR_T, BR_T, 0, s>>>(a);
  return cudaGetLastError();
}

template <int LK>
cudaError_t launch_brute_lk(const QueryArgs &a, int dp, int sms, cudaStream_t s) {
  if (dp == 8) return launch_brute_dp<LK, 8>(a, sms, s);
  if (dp == 16) return launch_brute_dp<LK, 16>(a, sms, s);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_cand_avg(const QueryArgs &a, int32_t *lpos, float *llb, int32_t *lcnt,
                            float *lub, int dp, cudaStream_t s) {
  if (a.nterm <= 0) return cudaSuccess;
  const int blocks = (a.nterm + BR_T - 1) / BR_T;
  switch (dp) {
    case 8: k_cand_avg<8><<<blocks, BR_T, 0, s>>>(a, lpos, llb, lcnt, lub); break;
    case 16: k_cand_avg<16><<<blocks, BR_T, 0, s>>>(a, lpos, llb, lcnt, lub); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// The exhaustive search of every terminal (closed-form linkages, FP32 bulk
// with FP64 re-score, one instance); pend_out must hold nterm entries, gu and
// gcnt too, glist GRAM_LIST per terminal, and ctr->npend must be 0.
cudaError_t launch_brute(const QueryArgs &a, int dp, int sms, cudaStream_t s) {
  if (a.nterm <= 0) return cudaSuccess;
  if (a.linkage == LK_WARD) return launch_brute_lk<LK_WARD>(a, dp, sms, s);
  if (a.linkage == LK_AVG2) return launch_brute_lk<LK_AVG2>(a, dp, sms, s);
  return cudaErrorInvalidValue;
}

}  // namespace hacg
