// Dense phase of average linkage (avg-1) and complete linkage: the whole matrix
// of pair distances once the active clusters fit.
//
// Section 5 keeps, per cluster, a table of up to s cached distances that
// Algorithm 5 updates by Lance-Williams after every merge.  When s reaches
// the number K of active clusters the table is the full K x K matrix, and no
// distance ever has to be evaluated twice.  On a GB300 that matrix fits for K
// in the tens of thousands (24 B per entry for average, 16 for complete):
//
//   * average linkage switches in mid-run: one all-pairs sweep of the points
//     fills the matrix: every pair of points in different clusters is visited
//     once (the points are laid out in cluster-contiguous segments in position
//     order, so a tile of 1,024 x 1,024 points covers a handful of cluster
//     pairs), and the sums of point distances are accumulated per cluster
//     pair.  Every such point pair enters exactly one later merge distance, so
//     the sweep does no work the exact answer does not need.  Complete linkage
//     would evaluate pairs that its range query prunes: it takes the matrix
//     only from the first round on, for runs of few points.  A run that starts
//     on the matrix fills it from the singletons (k_dense_single);
//   * every later round finds each terminal's nearest neighbour by a scan of
//     its row (Algorithm 2 without a range query: the matrix holds every
//     candidate), and after the merges a new, compacted matrix is written from
//     the old one (Table 2: D(A u B, C) is the weighted mean, or the maximum,
//     of D(A, C) and D(B, C));
//   * the chain update, reciprocal-pair filter, merges and compaction are the
//     ordinary round's kernels, so the rounds are those of Algorithm 1; below
//     DFIN_K clusters all rounds run in one launch (k_dense_finish).
//
// Exact sums.  Every entry is kept as the sum of its point distances in
// 128-bit fixed point (unit 2^e, chosen per instance so that (n/2)^2 times the
// largest point distance stays below 2^126 units), two 64-bit words, next to the
// mean distance that sum gives in FP64.  While the sweep or a re-score collects a
// sum it is four 32-bit limbs in 64-bit words, so that its atomic additions need
// no carry.  Integer addition is exact and associative, so:
//   * tiles can add into a cell with atomics in any order and the run is
//     deterministic;
//   * the Lance-Williams update of average linkage is the exact addition of
//     the sums (S(A u B, C) = S(A, C) + S(B, C)), with no rounding drift;
//   * in the FP64 mode a cell's sum is the exact sum of the FP64 point
//     distances of its pairs (each converts exactly), whatever the grouping,
//     so an FP64 re-score from the points in the FP32 mode reproduces the
//     FP64 mode's entry bit for bit, and both modes break exact ties alike.
//
// Precision.  FP64 mode: point distances in FP64, every entry exact.  FP32
// mode: the sweep uses the FP32 point copy and the stated error model of an
// FP32 point distance, |D32 - D| <= delta + rho D with rho = (d + 16) u + 32 u
// (FP32 partial sums of at most 32 terms), which sums and weighted means
// preserve; such an entry is an estimate.  A terminal's FP64 nearest
// neighbour is among the entries whose lower bound is within the least upper
// bound U; if that window holds estimates they are re-scored in FP64 from the
// points (GPU-wide) and the search is repeated, so the nearest neighbour,
// hence the tree, is the FP64 one.  A lone estimate whose bound is within
// 4e-6 relative keeps its upper bound as the height, as in the tree search.
#include "hac_impl.cuh"

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <utility>

namespace hacg {

namespace {

constexpr unsigned long long KINF_D = 0x7ff0000000000000ull;  // bits of +inf
constexpr unsigned long long SIGN = 0x8000000000000000ull;

// ---------------------------------------------------------------------------
// 128-bit fixed-point sums: value = (hi * 2^64 + lo) * 2^e; the top bit of hi
// marks an estimate (sums stay below 2^126 units, so it never carries)
// ---------------------------------------------------------------------------
constexpr unsigned long long TOP = 0x8000000000000000ull;

struct U128 {
  unsigned long long lo, hi;
};

// fixed-point value of v >= 0 (exact for v >= 2^(e+52), truncated below 2^e)
__device__ __forceinline__ U128 fx_of(double v, int e) {
  U128 r{0ull, 0ull};
  if (!(v > 0.0)) return r;
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  int E = (int)((bits >> 52) & 0x7ff);
  unsigned long long m = bits & 0xfffffffffffffull;
  if (E == 0)
    E = 1;  // subnormal
  else
    m |= 1ull << 52;
  int sh = E - 1075 - e;  // v = m * 2^(sh + e)
  if (sh > 74) sh = 74;   // cannot happen: every sum stays below 2^126 units
  if (sh >= 64) {
    r.hi = m << (sh - 64);
  } else if (sh > 0) {
    r.lo = m << sh;
    r.hi = m >> (64 - sh);
  } else if (sh == 0) {
    r.lo = m;
  } else if (sh > -64) {
    r.lo = m >> (-sh);
  }
  return r;
}

__device__ __forceinline__ void u128_add(U128 &a, const U128 &b) {
  const unsigned long long lo = a.lo + b.lo;
  a.hi += b.hi + (lo < a.lo ? 1ull : 0ull);
  a.lo = lo;
}

// A sum being collected is four 64-bit words, each the sum of one 32-bit limb of
// every addend (w0 + w1 2^32 + w2 2^64 + w3 2^96), so additions need no
// carries and go out as fire-and-forget atomics; 2^32 additions per word
// cannot overflow.  The estimate flag is the top bit of w3 (sums stay below
// 2^126 units, so w3 < 2^30).
constexpr int LIMBS = 4;

// the pair i < j of a k x k matrix in the packed upper triangle
__host__ __device__ __forceinline__ size_t tri(long long i, long long j, long long k) {
  return (size_t)(i * k - i * (i + 1) / 2 + (j - i - 1));
}

__device__ __forceinline__ void limbs_atomic(unsigned long long *w, const U128 &b) {
  if (!(b.lo | b.hi)) return;
  const unsigned long long l0 = b.lo & 0xffffffffull, l1 = b.lo >> 32;
  const unsigned long long l2 = b.hi & 0xffffffffull, l3 = b.hi >> 32;
  if (l0) atomicAdd(w, l0);
  if (l1) atomicAdd(w + 1, l1);
  if (l2) atomicAdd(w + 2, l2);
  if (l3) atomicAdd(w + 3, l3);
}

// the 128-bit value of four limb words (flag bit dropped) and the flag
__device__ __forceinline__ U128 limbs_value(const unsigned long long *w) {
  const unsigned long long w0 = w[0], w1 = w[1], w2 = w[2], w3 = w[3] & ~TOP;
  U128 r;
  r.lo = w0 + (w1 << 32);
  const unsigned long long c = r.lo < w0 ? 1ull : 0ull;
  r.hi = (w1 >> 32) + w2 + (w3 << 32) + c;
  return r;
}

// fixed-point value of a non-negative float (exact above 2^(e+23))
__device__ __forceinline__ U128 fx_of_f(float v, int e) {
  U128 r{0ull, 0ull};
  if (!(v > 0.f)) return r;
  const unsigned bits = __float_as_uint(v);
  int E = (int)((bits >> 23) & 0xff);
  unsigned long long m = bits & 0x7fffffu;
  if (E == 0)
    E = 1;
  else
    m |= 1ull << 23;
  int sh = E - 150 - e;  // v = m * 2^(sh + e)
  if (sh > 102) sh = 102;
  if (sh >= 64) {
    r.hi = m << (sh - 64);
  } else if (sh > 0) {
    r.lo = m << sh;
    r.hi = sh > 40 ? m >> (64 - sh) : 0ull;
  } else if (sh == 0) {
    r.lo = m;
  } else if (sh > -64) {
    r.lo = m >> (-sh);
  }
  return r;
}

__device__ __forceinline__ U128 u128_shfl_down(const U128 &v, int o) {
  return U128{__shfl_down_sync(0xffffffffu, v.lo, o), __shfl_down_sync(0xffffffffu, v.hi, o)};
}

__device__ __forceinline__ U128 u128_shfl_xor(const U128 &v, int o) {
  return U128{__shfl_xor_sync(0xffffffffu, v.lo, o), __shfl_xor_sync(0xffffffffu, v.hi, o)};
}

// A finished sum is two words (lo, hi), the estimate flag in the top bit of hi.
// The mean distance of an entry, one function everywhere so that equal sums
// and sizes give equal means, whichever cluster has which size: the 128-bit
// sum as the nearest FP64 number (to even), times 1 / size of the smaller
// cluster, times 1 / size of the other (reciprocals kept per matrix index: no
// FP64 division; one at a time, not their product, so that a sum that the sizes
// divide gives the whole quotient and true ties of lattice points stay ties);
// the sign bit set for an estimate.  The FP64 pipe (2 lanes per clock and SM)
// bounds every kernel that makes means, so the sum is converted by integer
// instructions and two FP64 multiplications are left: the matrix rebuild at
// 16,106 clusters took 1.90 ms with the seven FP64 instructions of two integer
// conversions and a scaled addition, 1.36 this way.
__device__ __noinline__ double sum_double_far(unsigned long long hi, unsigned long long lo, int e) {
  return ldexp((double)hi, 64 + e) + ldexp((double)lo, e);
}

__device__ __forceinline__ double sum_double(unsigned long long hi, unsigned long long lo, int e) {
  if (!(hi | lo)) return 0.0;
  // the leading 64 bits m (top bit set) and whether anything lies below them
  int up = 63 + e;  // exponent of the leading bit
  unsigned long long m = lo, rest = 0;
  if (hi) {
    const int sh = __clzll((long long)hi);
    m = sh ? (hi << sh) | (lo >> (64 - sh)) : hi;
    rest = lo << sh;
    up += 64 - sh;
  } else {
    const int sh = __clzll((long long)lo);
    m = lo << sh;
    up -= sh;
  }
  const int be = up + 1023;
  if (be < 1 || be > 2045) return sum_double_far(hi, lo, e);  // far outside any sensible scale
  unsigned long long r = m >> 11;
  const unsigned rem = (unsigned)(m & 0x7ff);
  r += rem > 0x400 || (rem == 0x400 && (rest || (r & 1)));
  // the leading bit adds 1 to the exponent; a carry out of the rounding too
  return __longlong_as_double((long long)(((unsigned long long)(be - 1) << 52) + r));
}

__device__ __forceinline__ double entry_mean(const U128 &v, int e, double inv_a, double inv_b) {
  // (ordered by integer comparisons: bits of positive numbers)
  const long long a = __double_as_longlong(inv_a), c = __double_as_longlong(inv_b);
  const double m = sum_double(v.hi & ~TOP, v.lo, e) * __longlong_as_double(max(a, c)) *
                   __longlong_as_double(min(a, c));
  const unsigned long long b = (unsigned long long)__double_as_longlong(m);
  return __longlong_as_double((long long)(v.hi & TOP ? (b | SIGN) : b));
}

// sum of two entries (the flags OR)
__device__ __forceinline__ U128 sum_add(const U128 &x, const U128 &y) {
  U128 r{x.lo, x.hi & ~TOP};
  u128_add(r, U128{y.lo, y.hi & ~TOP});
  r.hi |= (x.hi | y.hi) & TOP;
  return r;
}

// ---------------------------------------------------------------------------
// the all-pairs sweep
// ---------------------------------------------------------------------------
constexpr int DS_TPB = 256;  // threads per tile
constexpr int DS_CH = 256;   // columns per staged chunk
// FP32 sweep shape: rows per thread for d <= 8 (2 above), and the resident
// tiles per SM the register budget is cut for (the shape tuner's best at
// 10^6 points, 5-D: 4 and 4)
#ifndef HAC_DS_PPT8
#define HAC_DS_PPT8 4
#endif
#ifndef HAC_DS_MINB
#define HAC_DS_MINB 4
#endif
struct SweepArgs {
  const float *p32;
  const double *p64;
  const int32_t *plab;
  const int32_t *pos;  // matrix index (= position) of each cluster
  int64_t N;  // points in the layout
  int dk, e;
  // FP32 sweep: coordinates times scl = 2^k (exact), so that squared
  // distances flushed to zero by the square root (below 2^-126) are below
  // 2^(-126-2k) unscaled; sums of scaled distances convert with unit 2^es,
  // es = e + k, to the same fixed-point values
  float scl;
  int es;
  unsigned long long *sum;  // the packed upper triangle of sums (LIMBS words per pair)
  long long nb;             // blocks of TI points along each axis
  Counters *ctr;
};

__device__ __forceinline__ void tile_of(long long t, long long &bi, long long &bj) {
  long long j = (long long)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
  while (j * (j + 1) / 2 > t) --j;
  while ((j + 1) * (j + 2) / 2 <= t) ++j;
  bj = j;
  bi = t - j * (j + 1) / 2;
}

// Per chunk: segment starts of equal keys (cluster matrix indices) among the
// staged columns; returns the count, sstart[count] = cnt.
__device__ __forceinline__ int chunk_segments(const int *skey, int cnt, int *sstart, int *wtot) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const bool flag = t < cnt && (t == 0 || skey[t] != skey[t - 1]);
  const unsigned b = __ballot_sync(0xffffffffu, flag);
  if (lane == 0) wtot[w] = __popc(b);
  __syncthreads();
  int before = 0, total = 0;
  for (int i = 0; i < DS_TPB / 32; ++i) {
    before += i < w ? wtot[i] : 0;
    total += wtot[i];
  }
  if (flag) sstart[before + __popc(b & ((1u << lane) - 1u))] = t;
  if (t == 0) sstart[total] = cnt;
  __syncthreads();
  return total;
}

// Keys of a warp's rows are non-decreasing along the lanes, so equal keys
// form contiguous runs.  `same` holds, per step o = 1, 2, 4, 8, 16, whether
// lane + o has this lane's key; after seg_sum the first lane of each run
// holds the run's total.
__device__ __forceinline__ unsigned seg_mask(int k, int lane) {
  unsigned m = 0;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int k2 = __shfl_down_sync(0xffffffffu, k, 1 << i);
    if (lane + (1 << i) < 32 && k2 == k) m |= 1u << i;
  }
  return m;
}

__device__ __forceinline__ U128 seg_sum(U128 v, unsigned same) {
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const U128 v2 = u128_shfl_down(v, 1 << i);
    if ((same >> i) & 1u) u128_add(v, v2);
  }
  return v;
}

// Row layout of a warp: lane l holds PPT consecutive rows, r0 + l * PPT + r,
// so a lane's rows mostly share one key (cluster), and keys are
// non-decreasing along (lane, r).  Per lane: its head run (key of row 0), its
// tail run (key of row PPT - 1), and any runs wholly inside the lane.
struct RowKeys {
  int head, tail;
  unsigned same;  // seg_mask of the tail keys
  bool lead;      // first lane of its tail run
  bool absorbed;  // the head run continues the previous lane's tail run
  bool split;     // head != tail
};

// Row setup shared by both sweeps; returns whether all rows of the warp
// share one key.
template <int PPT>
__device__ __forceinline__ bool row_keys(const SweepArgs &a, long long r0, int lane,
                                         int (&krow)[PPT], RowKeys &rk, int &kfirst) {
#pragma unroll
  for (int r = 0; r < PPT; ++r) {
    const long long row = r0 + (long long)lane * PPT + r;
    krow[r] = row < a.N ? a.pos[a.plab[row]] : INT_MAX;
  }
  rk.head = krow[0];
  rk.tail = krow[PPT - 1];
  rk.split = rk.head != rk.tail;
  rk.same = seg_mask(rk.tail, lane);
  const int pt = __shfl_up_sync(0xffffffffu, rk.tail, 1);
  rk.lead = lane == 0 || pt != rk.tail;
  rk.absorbed = lane > 0 && rk.split && pt == rk.head;
  kfirst = __shfl_sync(0xffffffffu, rk.head, 0);
  const int klast = __shfl_sync(0xffffffffu, rk.tail, 31);
  return kfirst == klast;
}

// Flush one column segment (key qj) of every row: cell (key, qj) gets the
// sum of the rows with that key when key < qj (each unordered cluster pair
// once, its lower matrix index first).  Runs inside a lane are summed there;
// a head run that continues the previous lane's tail is handed to it; the
// tails are summed over each run of lanes by one segmented reduction.
template <int PPT>
__device__ __forceinline__ void flush(const SweepArgs &a, const U128 (&acc)[PPT],
                                      const int (&krow)[PPT], const RowKeys &rk, bool uniform,
                                      int qj, int lane) {
  if (uniform) {  // every row of the warp in one cluster
    if (!(krow[0] < qj)) return;
    U128 v = acc[0];
#pragma unroll
    for (int r = 1; r < PPT; ++r) u128_add(v, acc[r]);
#pragma unroll
    for (int o = 16; o; o >>= 1) u128_add(v, u128_shfl_xor(v, o));
    if (lane == 0) limbs_atomic(&a.sum[LIMBS * tri(krow[0], qj, a.dk)], v);
    return;
  }
  U128 vh{0ull, 0ull}, vt{0ull, 0ull};
#pragma unroll
  for (int r = 0; r < PPT; ++r) {
    if (krow[r] == rk.tail)
      u128_add(vt, acc[r]);
    else if (krow[r] == rk.head)
      u128_add(vh, acc[r]);
  }
  if (rk.split) {
    // runs wholly inside this lane (a cluster of fewer than PPT points here)
    int k = -1;
    U128 m{0ull, 0ull};
#pragma unroll
    for (int r = 0; r < PPT; ++r) {
      const int kr = krow[r];
      if (kr == rk.head || kr == rk.tail) continue;
      if (kr != k) {
        if (k >= 0 && k < qj) limbs_atomic(&a.sum[LIMBS * tri(k, qj, a.dk)], m);
        k = kr;
        m = U128{0ull, 0ull};
      }
      u128_add(m, acc[r]);
    }
    if (k >= 0 && k < qj) limbs_atomic(&a.sum[LIMBS * tri(k, qj, a.dk)], m);
  }
  // the next lane's head joins this tail when it continues the run
  const U128 nh = u128_shfl_down(vh, 1);
  const bool nabs = __shfl_down_sync(0xffffffffu, rk.absorbed, 1);
  if (lane < 31 && nabs) u128_add(vt, nh);
  if (rk.split && !rk.absorbed && rk.head < qj)
    limbs_atomic(&a.sum[LIMBS * tri(rk.head, qj, a.dk)], vh);
  vt = seg_sum(vt, rk.same);
  if (rk.lead && rk.tail < qj) limbs_atomic(&a.sum[LIMBS * tri(rk.tail, qj, a.dk)], vt);
}

// FP32 sweep, specialised on the true dimension D (rows of stride DP
// floats), PPT rows per thread; a tile is TI x TI points, TI = 256 * PPT.
// Two of a thread's rows share each f32x2 word (one coordinate of each) and
// every staged column is duplicated into both halves, so one packed subtract
// and one packed multiply-add advance two point pairs by one coordinate.  Per
// row and column segment: FP32 partial sums of at most 32 terms (two rows' sums
// per packed word), each converted to fixed point exactly and added as integers
// (no FP64 work).  Columns are staged padded to whole 16-byte words: 3 instead of
// 5 loads and 2 instead of 4 additions per column at d = 5 took the sweep of 10^6
// points from 220 to 206 ms (17 flops per pair: 41 TFLOP/s of the 80 measured).
template <int D, int DP, int PPT>
__global__ void __launch_bounds__(DS_TPB, HAC_DS_MINB) k_dense_sweep32(SweepArgs a) {
  constexpr int TI = DS_TPB * PPT, NP = PPT / 2;
  constexpr int DE = (D + 1) & ~1;  // staged columns are read 16 bytes at a time
  __shared__ __align__(16) unsigned long long sy[DS_CH * DE];
  __shared__ int skey[DS_CH];
  __shared__ int sstart[DS_CH + 1];
  __shared__ int wtot[DS_TPB / 32];
  long long bi, bj;
  tile_of(blockIdx.x + (long long)gridDim.x * blockIdx.y, bi, bj);
  if (bi >= a.nb || bj >= a.nb) return;  // uniform over the block
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long r0 = bi * TI + (long long)w * 32 * PPT;
  unsigned long long x[NP][D];
  int krow[PPT];
  RowKeys rk;
  int kfirst;
  const bool uniform = row_keys<PPT>(a, r0, lane, krow, rk, kfirst);
#pragma unroll
  for (int h = 0; h < NP; ++h) {
    const long long ra = r0 + (long long)lane * PPT + 2 * h, rb = ra + 1;
#pragma unroll
    for (int k = 0; k < D; ++k)
      x[h][k] = f2_pack(ra < a.N ? a.p32[(size_t)ra * DP + k] * a.scl : 0.f,
                        rb < a.N ? a.p32[(size_t)rb * DP + k] * a.scl : 0.f);
  }
  unsigned long long pairs = 0;
  for (int ch = 0; ch < PPT; ++ch) {  // TI columns in chunks of DS_CH
    const long long c0 = bj * TI + (long long)ch * DS_CH;
    if (c0 >= a.N) break;  // uniform
    const int cnt = (int)min((long long)DS_CH, a.N - c0);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt * D; i += DS_TPB) {
      const int c = i / D, k = i - c * D;
      const float y = a.p32[(size_t)(c0 + c) * DP + k] * a.scl;
      sy[c * DE + k] = f2_pack(y, y);
    }
    if (threadIdx.x < DS_CH)
      skey[threadIdx.x] = threadIdx.x < cnt ? a.pos[a.plab[c0 + threadIdx.x]] : -1;
    __syncthreads();
    const int nseg = chunk_segments(skey, cnt, sstart, wtot);
    for (int sg = 0; sg < nseg; ++sg) {
      const int cb = sstart[sg], ce = sstart[sg + 1];
      const int qj = skey[cb];
      if (qj <= kfirst) continue;  // no row of this warp pairs with it (uniform)
      U128 acc[PPT];
#pragma unroll
      for (int r = 0; r < PPT; ++r) acc[r] = U128{0ull, 0ull};
      for (int c1 = cb; c1 < ce; c1 += 32) {
        const int c2 = min(c1 + 32, ce);
        unsigned long long part[NP];  // two rows' sums per word
#pragma unroll
        for (int h = 0; h < NP; ++h) part[h] = 0ull;
#pragma unroll 2
        for (int c = c1; c < c2; ++c) {
          unsigned long long y[DE];
#pragma unroll
          for (int k = 0; k < DE; k += 2) {
            const ulonglong2 w = *(const ulonglong2 *)&sy[c * DE + k];
            y[k] = w.x;
            y[k + 1] = w.y;
          }
#pragma unroll
          for (int h = 0; h < NP; ++h) {
            unsigned long long t = f2_sub(x[h][0], y[0]);
            unsigned long long d2 = f2_mul(t, t);
#pragma unroll
            for (int k = 1; k < D; ++k) {
              t = f2_sub(x[h][k], y[k]);
              d2 = f2_fma(t, t, d2);
            }
            float s0, s1;
            f2_unpack(d2, s0, s1);
            part[h] = f2_add(part[h], f2_pack(sqrt_approx_ftz(s0), sqrt_approx_ftz(s1)));
          }
        }
#pragma unroll
        for (int h = 0; h < NP; ++h) {
          float p0, p1;
          f2_unpack(part[h], p0, p1);
          u128_add(acc[2 * h], fx_of_f(p0, a.es));
          u128_add(acc[2 * h + 1], fx_of_f(p1, a.es));
        }
      }
      int below = 0;
#pragma unroll
      for (int r = 0; r < PPT; ++r) below += krow[r] < qj;
      pairs += (unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)below) * (ce - cb);
      flush<PPT>(a, acc, krow, rk, uniform, qj, lane);
    }
  }
  if (lane == 0 && pairs) atomicAdd(&a.ctr->dense_pp, pairs);
}

// FP64 sweep: the same tiles, FP64 coordinates, specialised on the true
// dimension too (the FP64 pipe bounds it: 2 D operations and a square root per
// pair); every point distance is added to the row's 128-bit sum exactly.
template <int D, int DP, int PPT>
__global__ void __launch_bounds__(DS_TPB) k_dense_sweep64(SweepArgs a) {
  constexpr int TI = DS_TPB * PPT;
  __shared__ double sy[DS_CH * D];
  __shared__ int skey[DS_CH];
  __shared__ int sstart[DS_CH + 1];
  __shared__ int wtot[DS_TPB / 32];
  long long bi, bj;
  tile_of(blockIdx.x + (long long)gridDim.x * blockIdx.y, bi, bj);
  if (bi >= a.nb || bj >= a.nb) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long r0 = bi * TI + (long long)w * 32 * PPT;
  double x[PPT][D];
  int krow[PPT];
  RowKeys rk;
  int kfirst;
  const bool uniform = row_keys<PPT>(a, r0, lane, krow, rk, kfirst);
#pragma unroll
  for (int r = 0; r < PPT; ++r) {
    const long long row = r0 + (long long)lane * PPT + r;
#pragma unroll
    for (int k = 0; k < D; ++k) x[r][k] = row < a.N ? a.p64[(size_t)row * DP + k] : 0.0;
  }
  unsigned long long pairs = 0;
  for (int ch = 0; ch < PPT; ++ch) {
    const long long c0 = bj * TI + (long long)ch * DS_CH;
    if (c0 >= a.N) break;
    const int cnt = (int)min((long long)DS_CH, a.N - c0);
    __syncthreads();
    for (int i = threadIdx.x; i < cnt * D; i += DS_TPB) {
      const int c = i / D, k = i - c * D;
      sy[i] = a.p64[(size_t)(c0 + c) * DP + k];
    }
    if (threadIdx.x < DS_CH)
      skey[threadIdx.x] = threadIdx.x < cnt ? a.pos[a.plab[c0 + threadIdx.x]] : -1;
    __syncthreads();
    const int nseg = chunk_segments(skey, cnt, sstart, wtot);
    for (int sg = 0; sg < nseg; ++sg) {
      const int cb = sstart[sg], ce = sstart[sg + 1];
      const int qj = skey[cb];
      if (qj <= kfirst) continue;
      U128 acc[PPT];
#pragma unroll
      for (int r = 0; r < PPT; ++r) acc[r] = U128{0ull, 0ull};
      for (int c = cb; c < ce; ++c) {
        const double *y = sy + c * D;
#pragma unroll
        for (int r = 0; r < PPT; ++r) {
          double d2 = 0.0;
#pragma unroll
          for (int k = 0; k < D; ++k) {
            const double t = x[r][k] - y[k];
            d2 = fma(t, t, d2);
          }
          u128_add(acc[r], fx_of(sqrt(d2), a.e));
        }
      }
      int below = 0;
#pragma unroll
      for (int r = 0; r < PPT; ++r) below += krow[r] < qj;
      pairs += (unsigned long long)__reduce_add_sync(0xffffffffu, (unsigned)below) * (ce - cb);
      flush<PPT>(a, acc, krow, rk, uniform, qj, lane);
    }
  }
  if (lane == 0 && pairs) atomicAdd(&a.ctr->dense_pp, pairs);
}

// ---------------------------------------------------------------------------
// building the matrix
// ---------------------------------------------------------------------------
// The matrix is indexed by position in the active order, so a row scan reads
// one contiguous row.  Means are kept as the full square (row stride dld),
// sums as the packed upper triangle.  32 x 32 tiles of the upper triangle with
// their mirror tile go through shared memory, so every global access is a row
// segment; threads are 32 x 8.
constexpr int FT_Y = 8;

__device__ __forceinline__ bool fin_tile(int K, long long &ti, long long &tj) {
  // consecutive blocks take consecutive tiles of one tile row, so the rows of
  // sums and means in flight together are long.  One warp works the tile out,
  // not all eight: the FP64 square root in tile_of helped to keep the FP64 pipe
  // 63 % busy in the fill (rebuilds of an average run of 20,001 10-D points 8.2
  // ms, 7.3 this way; its fill 2.9, 2.7).
  __shared__ long long s_tile[2];
  const int nt = (K + 31) / 32;
  if (threadIdx.y == 0) {
    long long bi, bj;
    tile_of(blockIdx.x + (long long)gridDim.x * blockIdx.y, bi, bj);
    if (threadIdx.x == 0) {
      s_tile[0] = nt - 1 - bj;
      s_tile[1] = nt - 1 - bi;
    }
  }
  __syncthreads();
  ti = s_tile[0];
  tj = s_tile[1];
  return ti >= 0 && tj >= 0;
}

// upper tile in Mv (row k, column tx) -> both triangles of the mean matrix
__device__ __forceinline__ void fin_store(double *mat, int ld, int K, long long ti, long long tj,
                                          double (*Mv)[33]) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  __syncthreads();
  for (int k = ty; k < 32; k += FT_Y) {
    const long long i = ti * 32 + k, j = tj * 32 + tx;
    if (i < K && j < K)  // diagonal tile: the lower cells take the upper cells' means
      mat[(size_t)i * ld + j] = ti == tj && i > j ? Mv[tx][k] : Mv[k][tx];
    if (ti != tj) {  // mirror tile: row tj*32+k, column ti*32+tx = upper cell (tx, k)
      const long long i2 = tj * 32 + k, j2 = ti * 32 + tx;
      if (i2 < K && j2 < K) mat[(size_t)i2 * ld + j2] = Mv[tx][k];
    }
  }
}

__device__ __forceinline__ U128 sum_at(const unsigned long long *sum, int i, int j, int K) {
  const ulonglong2 w = __ldcg((const ulonglong2 *)sum + (i < j ? tri(i, j, K) : tri(j, i, K)));
  return U128{w.x, w.y};
}

// the sweep's limb sums as two-word sums, in another buffer
__global__ void k_dense_pack(const unsigned long long *limb, unsigned long long *sum, size_t cells,
                             bool est) {
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < cells;
       t += (size_t)gridDim.x * blockDim.x) {
    const U128 v = limbs_value(limb + LIMBS * t);
    ((ulonglong2 *)sum)[t] = make_ulonglong2(v.lo, v.hi | (est ? TOP : 0ull));
  }
}

// means of the packed sums (+inf on the diagonal)
__global__ void __launch_bounds__(32 * FT_Y) k_dense_mean(State s, int K) {
  __shared__ double Mv[32][33];
  long long ti, tj;
  if (!fin_tile(K, ti, tj)) return;
  for (int k = threadIdx.y; k < 32; k += FT_Y) {
    const int i = (int)ti * 32 + k, j = (int)tj * 32 + threadIdx.x;
    double v = __longlong_as_double((long long)KINF_D);
    if (i < j && j < K) v = entry_mean(sum_at(s.dsum, i, j, K), s.dexp, s.dinv[i], s.dinv[j]);
    Mv[k][threadIdx.x] = v;
  }
  fin_store(s.dmat, s.dld, K, ti, tj, Mv);
}

__global__ void k_dense_init(State s, const int32_t *order, int K, unsigned long long pairs) {
  if (blockIdx.x == 0 && threadIdx.x == 0) s.ctr->dense_pp += pairs;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < K; p += gridDim.x * blockDim.x)
    s.dinv[p] = 1.0 / (double)s.csize[order[p]];
}

// FP64 distance of a pair whose FP32 distance is zero (rare: kept out of line)
__device__ __noinline__ double dist64(const double *x, const double *y, int d) {
  double s = 0.0;
  for (int c = 0; c < d; ++c) {
    const double t = x[c] - y[c];
    s = fma(t, t, s);
  }
  return sqrt(s);
}

// The matrix of K singletons, straight from the points (position p is point p
// of the layout): one thread per pair, no sums to collect by atomics.  The
// distances are those of the sweeps (FP32: scaled coordinates, for average the
// flush-to-zero root; FP64: the same fma chain).  Bound by the 24-32 B written per pair, or
// in FP64 by the square roots; the segmented sweep, which flushes every column
// of every row through atomics when each point is a cluster of its own, took
// 11 ms with its last pass at 20,001 points in 10-D, this 2.7.
template <int LK, int DP, int F32>
__global__ void __launch_bounds__(32 * FT_Y) k_dense_single(State s, const float *p32,
                                                             const double *p64, int K, float scl,
                                                             int es, float inv_scl) {
  using T = typename std::conditional<F32 != 0, float, double>::type;
  __shared__ double Mv[32][33];
  __shared__ T sx[32][DP + 1];
  long long ti, tj;
  if (!fin_tile(K, ti, tj)) return;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int t = ty * 32 + tx; t < 32 * DP; t += 32 * FT_Y) {
    const int r = t / DP, k = t - r * DP;
    const long long i = ti * 32 + r;
    T v = 0;
    if (i < K) v = F32 ? (T)(p32[(size_t)i * DP + k] * scl) : (T)p64[(size_t)i * DP + k];
    sx[r][k] = v;
  }
  const int j = (int)tj * 32 + tx;
  T y[DP];
#pragma unroll
  for (int k = 0; k < DP; ++k) {
    y[k] = 0;
    if (j < K) y[k] = F32 ? (T)(p32[(size_t)j * DP + k] * scl) : (T)p64[(size_t)j * DP + k];
  }
  __syncthreads();
  for (int k = ty; k < 32; k += FT_Y) {
    const int i = (int)ti * 32 + k;
    double v = __longlong_as_double((long long)KINF_D);
    if (i < j && j < K) {
      T d2 = 0;
#pragma unroll
      for (int c = 0; c < DP; ++c) {
        if (c < s.d) {
          const T t = sx[k][c] - y[c];
          d2 = fma(t, t, d2);
        }
      }
      // a zero FP32 distance (duplicates, mostly) is settled in FP64 at once:
      // as estimates, large groups of duplicates would all be re-scored
      double z = 0.0;
      const bool zero = F32 && d2 == (T)0;
      if (zero) z = dist64(p64 + (size_t)i * DP, p64 + (size_t)j * DP, s.d);
      if (LK == LK_COMPLETE) {
        if (zero) {
          v = z;
        } else if (F32) {
          // the rounded root, as the evaluations of the searches take it; back to
          // unscaled units (a power of two: exact)
          const double m = (double)sqrtf((float)d2) * (double)inv_scl;
          v = __longlong_as_double((long long)((unsigned long long)__double_as_longlong(m) | SIGN));
        } else {
          v = sqrt((double)d2);
        }
      } else {
        U128 u = zero ? fx_of(z, s.dexp)
                 : F32 ? fx_of_f(sqrt_approx_ftz((float)d2), es)
                       : fx_of(sqrt((double)d2), s.dexp);
        if (F32 && !zero) u.hi |= TOP;
        ((ulonglong2 *)s.dsum)[tri(i, j, K)] = make_ulonglong2(u.lo, u.hi);
        v = entry_mean(u, s.dexp, s.dinv[i], s.dinv[j]);
      }
    }
    Mv[k][tx] = v;
  }
  fin_store(s.dmat, s.dld, K, ti, tj, Mv);
}

// ---------------------------------------------------------------------------
// nearest neighbours on the matrix: one warp per terminal, a scan of its row
// ---------------------------------------------------------------------------
struct NNArgs {
  const double *dmat;
  int ld, K, nlist;
  const int32_t *order, *pos, *list;
  // FP32 mode: error model of an estimate x of the FP64 value D,
  // |x - D| <= delta + rho D + eta; eta (absolute) covers the sums' fixed-
  // point truncation (below one unit 2^e per partial sum, on both sides)
  // and the square roots' flush of squared distances below 2^-126 (scaled)
  double delta, rho, eta;
  // FP32 mode with delta = 0: the bounds as steps of the FP64 bit pattern
  // (adding N ulps to a non-negative double multiplies it by at least
  // 1 + N 2^-53): for x >= m0 (so eta <= 2^-30 x) up = x + nu ulps >=
  // (x + eta) / (1 - rho) and lo = x - nl ulps <= (x - eta) / (1 + rho) (nl
  // doubled for a step down across a power of two); an estimate below m0
  // spans [0, m0up] (m0up = 2 m0 >= its upper bound)
  unsigned long long nu, nl, m0, m0up;
  double *Ekey;
  int32_t *Ecid;
  int32_t *drq_a, *drq_b;
  int drq_cap;
  int32_t *pend_out;
  Counters *ctr;
};

__device__ __forceinline__ bool kless_d(unsigned long long k1, int c1, unsigned long long k2,
                                        int c2) {
  return k1 < k2 || (k1 == k2 && c1 < c2);
}

__device__ __forceinline__ void warp_argmin_kc(unsigned long long &k, int &c) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, k, o);
    const int c2 = __shfl_xor_sync(0xffffffffu, c, o);
    if (kless_d(k2, c2, k, c)) {
      k = k2;
      c = c2;
    }
  }
}

__device__ __forceinline__ unsigned long long warp_min_u(unsigned long long v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w < v ? w : v;
  }
  return v;
}

// Upper bound of an estimate, and the largest estimate whose lower bound is
// within U.  Both are monotone in the estimate, so a scan only needs the
// least estimate and the least exact entry to know U, and tests the window
// by one integer comparison (no FP64 arithmetic per entry).
//   F32 == 2: integer steps (delta = 0)
//   F32 == 1: FP64 arithmetic: (x - delta - eta) / (1 + rho) <= D <=
//   (x + delta + eta) / (1 - rho), widened by 1e-12 for the rounding of these
//   operations; x - delta - eta rounds by up to 2^-52 max(x, dl), so the
//   lower bound subtracts dl (1 + 2^-50).
template <int F32>
__device__ __forceinline__ unsigned long long est_up(const NNArgs &a, unsigned long long m) {
  if (F32 == 2) return m < a.m0 ? a.m0up : m + a.nu;
  const double up_f = (1.0 + 1e-12) / (1.0 - a.rho);
  return (unsigned long long)__double_as_longlong(
      (__longlong_as_double((long long)m) + (a.delta + a.eta)) * up_f);
}
template <int F32>
__device__ __forceinline__ unsigned long long est_window(const NNArgs &a, unsigned long long U) {
  if (U >= KINF_D) return U;
  if (F32 == 2) return max(U + a.nl, a.m0);
  const double dlo = (a.delta + a.eta) * (1.0 + 0x1p-50), lo_f = (1.0 - 1e-12) / (1.0 + a.rho);
  // max(m - dlo, 0) lo_f <= U  <=>  m <= U / lo_f + dlo, rounded up
  return (unsigned long long)__double_as_longlong(
      (__longlong_as_double((long long)U) / lo_f + dlo) * (1.0 + 1e-12));
}

// What one scan of a row found (warp-uniform): `kind` 1 = decided (key bits and
// cid), 0 = estimates within `win` need their FP64 values, -1 = no candidate
struct RowNN {
  int kind, cid;
  unsigned long long key, win;
};

constexpr int NN_U = 4;  // 16-byte loads of the row in flight per lane

// `order` gives cids by position; the row has K entries, +inf for the row's own
template <int F32>
__device__ __forceinline__ RowNN row_scan(const NNArgs &a, const double *row, const int32_t *order,
                                          int K, int lane) {
  // exact entries: least (key, cid); estimates: the two least and the least's position
  unsigned long long xk = KINF_D, e1 = ~0ull, e2 = ~0ull;
  int xp = -1, p1 = -1;
  for (int p0 = 0; p0 < K; p0 += 64 * NN_U) {
    ulonglong2 v[NN_U];
#pragma unroll
    for (int u = 0; u < NN_U; ++u) {
      const int p = p0 + u * 64 + 2 * lane;
      v[u] = make_ulonglong2(KINF_D, KINF_D);
      if (p < K) {  // rows are padded: the second entry may lie past K
        v[u] = __ldcg((const ulonglong2 *)(row + p));
        if (p + 1 >= K) v[u].y = KINF_D;
      }
    }
#pragma unroll
    for (int u = 0; u < NN_U; ++u)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int p = p0 + u * 64 + 2 * lane + h;
        const unsigned long long x = h ? v[u].y : v[u].x;
        if (F32 && (x & SIGN)) {
          const unsigned long long m = x & ~SIGN;
          if (m < e1) {
            e2 = e1;
            e1 = m;
            p1 = p;
          } else if (m < e2) {
            e2 = m;
          }
        } else if (x < xk || (x == xk && xp >= 0 && order[p] < order[xp])) {
          xk = x;
          xp = p;
        }
      }
  }
  RowNN r;
  r.win = 0;
  int xc = xp >= 0 ? order[xp] : INT_MAX;
  warp_argmin_kc(xk, xc);
  r.key = xk;
  r.cid = xc;
  r.kind = xc == INT_MAX ? -1 : 1;
  if (!F32) return r;
  const unsigned long long em = warp_min_u(e1);
  if (em == ~0ull) return r;  // no estimates in the row
  const unsigned long long up = est_up<F32>(a, em);
  const unsigned long long U = up < xk ? up : xk;
  r.win = est_window<F32>(a, U);
  if (em > r.win) return r;  // the least exact entry wins
  const unsigned holder = __ballot_sync(0xffffffffu, e1 <= r.win);
  const unsigned more = __ballot_sync(0xffffffffu, e2 <= r.win);
  r.kind = 0;
  if (xk <= U || more || __popc(holder) != 1) return r;
  // the lone candidate is an estimate: its upper bound stands in for the
  // FP64 value when the stated bound is within 4e-6 relative (F32 == 2:
  // checked by the host, unless the absolute term dominates, below m0)
  bool fine = em >= a.m0;
  if (F32 == 1) {
    const double x = __longlong_as_double((long long)em);
    fine = (a.delta + a.eta) + a.rho * x <= 4e-6 * x;
  }
  if (!fine) return r;
  r.kind = 1;
  r.key = up;
  r.cid = order[__shfl_sync(0xffffffffu, p1, __ffs(holder) - 1)];
  return r;
}

template <int F32>
__global__ void __launch_bounds__(256) k_dense_nn(NNArgs a) {
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  unsigned long long tests = 0;
  for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < a.nlist; t += nw) {
    const int ci = a.list[t];
    const int qi = a.pos[ci];
    const double *row = a.dmat + (size_t)qi * a.ld;
    tests += (unsigned long long)(a.K - 1);
    const RowNN r = row_scan<F32>(a, row, a.order, a.K, lane);
    if (r.kind) {
      if (lane == 0) {
        a.Ekey[ci] = __longlong_as_double((long long)r.key);
        a.Ecid[ci] = r.kind < 0 ? -1 : r.cid;
        if (r.kind < 0) atomicOr(&a.ctr->err, ERR_NO_NN);
      }
      continue;
    }
    // estimates in the window: re-score them in FP64
    for (int p = lane; p < a.K; p += 32) {
      const unsigned long long x = (unsigned long long)__double_as_longlong(row[p]);
      if (!(x & SIGN) || (x & ~SIGN) > r.win) continue;
      // a full list counts no further: 2^31 estimates can lie in the windows of
      // 46,341 terminals, and a wrapped counter would pass as an index
      if (*(volatile int32_t *)&a.ctr->nrq >= a.drq_cap) break;
      const int q = atomicAdd(&a.ctr->nrq, 1);
      if (q < a.drq_cap) {
        a.drq_a[q] = min(qi, p);
        a.drq_b[q] = max(qi, p);
      }
    }
    if (lane == 0) a.pend_out[atomicAdd(&a.ctr->npend, 1)] = ci;
  }
  if (lane == 0 && tests) atomicAdd(&a.ctr->ltests, tests);
}

// ---------------------------------------------------------------------------
// FP64 re-score of listed pairs from the points (GPU-wide)
// ---------------------------------------------------------------------------
constexpr int RQ_TPB = 256;   // rows (points of the first cluster) per tile
constexpr int RQ_COLS = 1024; // points of the second cluster per tile
constexpr int RQ_CH = 128;    // staged per chunk

__global__ void k_drq_count(State s, const int32_t *order, int m) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const int A = order[s.drq_a[i]], B = order[s.drq_b[i]];
    const long long na = s.csize[A], nb = s.csize[B];
    s.drq_pre[i] = (int32_t)(((na + RQ_TPB - 1) / RQ_TPB) * ((nb + RQ_COLS - 1) / RQ_COLS));
  }
}

// exclusive scan of m tile counts into drq_pre (one block; total at [m])
__global__ void k_drq_scan(State s, int m) {
  __shared__ long long part[1024];
  const int t = threadIdx.x, T = blockDim.x;
  const int per = (m + T - 1) / T, b0 = t * per;
  long long sum = 0;
  for (int i = 0; i < per; ++i)
    if (b0 + i < m) sum += s.drq_pre[b0 + i];
  part[t] = sum;
  __syncthreads();
  if (t == 0) {
    long long run = 0;
    for (int i = 0; i < T; ++i) {
      const long long v = part[i];
      part[i] = run;
      run += v;
    }
    s.drq_pre[m] = (int32_t)min(run, (long long)INT_MAX);
    if (run > INT_MAX) atomicOr(&s.ctr->err, ERR_WINDOW);  // far beyond any real queue
  }
  __syncthreads();
  long long run = part[t];
  for (int i = 0; i < per; ++i)
    if (b0 + i < m) {
      const long long v = s.drq_pre[b0 + i];
      s.drq_pre[b0 + i] = (int32_t)run;
      run += v;
    }
}

template <int LK, int DP>
__global__ void __launch_bounds__(RQ_TPB) k_drq_eval(State s, const int32_t *order, int m, int cur) {
  __shared__ double sy[RQ_CH * DP];
  __shared__ unsigned long long rlo[RQ_TPB / 32], rhi[RQ_TPB / 32];
  const int total = s.drq_pre[m];
  const double *P = s.p64[cur];
  const int32_t *seg = s.seg[cur];
  for (int t = blockIdx.x; t < total; t += gridDim.x) {
    int lo = 0, hi = m - 1;  // last i with pre[i] <= t
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s.drq_pre[mid] <= t) lo = mid; else hi = mid - 1;
    }
    const int i = lo;
    const int A = order[s.drq_a[i]], B = order[s.drq_b[i]];
    const int na = s.csize[A], nb = s.csize[B];
    const int tbn = (nb + RQ_COLS - 1) / RQ_COLS;
    const int j = t - s.drq_pre[i];
    const int ta = j / tbn, tb = j - ta * tbn;
    const int row = ta * RQ_TPB + threadIdx.x;
    double x[DP];
    const bool act = row < na;
#pragma unroll
    for (int k = 0; k < DP; ++k) x[k] = act ? P[(size_t)(seg[A] + row) * DP + k] : 0.0;
    U128 acc{0ull, 0ull};
    double mx = 0.0;
    const int cbeg = tb * RQ_COLS, cend = min(nb, cbeg + RQ_COLS);
    for (int c0 = cbeg; c0 < cend; c0 += RQ_CH) {
      const int cnt = min(RQ_CH, cend - c0);
      __syncthreads();
      for (int q = threadIdx.x; q < cnt * DP; q += RQ_TPB)
        sy[q] = P[(size_t)(seg[B] + c0) * DP + q];
      __syncthreads();
      if (act)
        for (int c = 0; c < cnt; ++c) {
          double d2 = 0.0;
#pragma unroll
          for (int k = 0; k < DP; ++k) {
            const double u = x[k] - sy[c * DP + k];
            d2 = fma(u, u, d2);
          }
          if (LK == LK_COMPLETE)
            mx = fmax(mx, d2);
          else
            u128_add(acc, fx_of(sqrt(d2), s.dexp));  // exactly as the FP64 sweep
        }
    }
    if (LK == LK_COMPLETE) acc.lo = (unsigned long long)__double_as_longlong(mx);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const U128 w = u128_shfl_xor(acc, o);
      if (LK == LK_COMPLETE)
        acc.lo = max(acc.lo, w.lo);  // bits of non-negative doubles
      else
        u128_add(acc, w);
    }
    if ((threadIdx.x & 31) == 0) {
      rlo[threadIdx.x >> 5] = acc.lo;
      rhi[threadIdx.x >> 5] = acc.hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      U128 v{0ull, 0ull};
      for (int w = 0; w < RQ_TPB / 32; ++w) {
        if (LK == LK_COMPLETE)
          v.lo = max(v.lo, rlo[w]);
        else
          u128_add(v, U128{rlo[w], rhi[w]});
      }
      if (LK == LK_COMPLETE)
        atomicMax(&s.drq_acc[LIMBS * (size_t)i], v.lo);
      else
        limbs_atomic(&s.drq_acc[LIMBS * (size_t)i], v);
      const long long rows = min(RQ_TPB, na - ta * RQ_TPB);
      atomicAdd(&s.ctr->dense_rq_pp, (unsigned long long)(rows * (cend - cbeg)));
    }
  }
}

// the re-scored values replace both entries (exact: no flag)
template <int LK>
__global__ void k_drq_fin(State s, int m) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x) {
    const int qa = s.drq_a[i], qb = s.drq_b[i];  // qa < qb
    const unsigned long long *w = s.drq_acc + LIMBS * (size_t)i;
    double v;
    if (LK == LK_COMPLETE) {
      v = sqrt(__longlong_as_double((long long)w[0]));
    } else {
      const U128 u = limbs_value(w);
      ((ulonglong2 *)s.dsum)[tri(qa, qb, s.dk)] = make_ulonglong2(u.lo, u.hi);
      v = entry_mean(u, s.dexp, s.dinv[qa], s.dinv[qb]);
    }
    s.dmat[(size_t)qa * s.dld + qb] = v;
    s.dmat[(size_t)qb * s.dld + qa] = v;
  }
}

// ---------------------------------------------------------------------------
// Lance-Williams update of the matrix after the round's merges.  Every merged
// row touches every column, and 10-20 % of the clusters merge in a round, so
// the next round's matrix is written anew over the compacted positions
// instead of patching rows and columns in place: each old entry is read once
// and each new one written once, all in row segments (average: 8 K^2 B of
// sums read, 8 K'^2 B of sums and 8 K'^2 B of means written), and later scans
// read no dead columns.  Patching in place (scattered column writes and
// packed-column reads) took 18.9 ms at 20,001 points in 10-D, this 7.3 with
// the compactions of the lists; the row scans fell from 14.6 to 7.5 ms.
// Average linkage: the sum of A u B with C is the sum of A's and B's (exact),
// the mean follows from the new sizes.  Complete: the larger entry.
// ---------------------------------------------------------------------------

// old positions of every new position's cluster (dma) and of the cluster that
// it merged with (dmb, -1 = none), and its 1 / size.  After the compaction:
// pos of a retired cid is still its old position.
__global__ void k_dense_map(State s, const int32_t *order_old, int Kold, int round) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < Kold; p += gridDim.x * blockDim.x) {
    const int c = order_old[p];
    if (!s.alive[c]) continue;
    const int q = s.pos[c];
    s.dma[q] = p;
    s.dmb[q] = s.mround[c] == round ? s.pos[s.partner[c]] : -1;
    s.dinv[q] = 1.0 / (double)s.csize[c];
  }
}

// the sum of new entry (a u b, c u d), b and d -1 if that side did not merge
__device__ __forceinline__ U128 sum_new(const unsigned long long *sum, int a, int b, int c, int d,
                                        int Kold) {
  U128 v = sum_at(sum, a, c, Kold);
  if (b >= 0) v = sum_add(v, sum_at(sum, b, c, Kold));
  if (d >= 0) {
    v = sum_add(v, sum_at(sum, a, d, Kold));
    if (b >= 0) v = sum_add(v, sum_at(sum, b, d, Kold));
  }
  return v;
}

// the larger of two entries; an estimate if either is one
__device__ __forceinline__ unsigned long long ent_max(unsigned long long x, unsigned long long y) {
  const unsigned long long mx = x & ~SIGN, my = y & ~SIGN;
  return (mx > my ? mx : my) | ((x | y) & SIGN);
}
__device__ __forceinline__ unsigned long long max_new(const double *mat, int ld, int a, int b, int c,
                                                      int d) {
  const unsigned long long *M = (const unsigned long long *)mat;
  unsigned long long v = __ldcg(M + (size_t)a * ld + c);
  if (b >= 0) v = ent_max(v, __ldcg(M + (size_t)b * ld + c));
  if (d >= 0) {
    v = ent_max(v, __ldcg(M + (size_t)a * ld + d));
    if (b >= 0) v = ent_max(v, __ldcg(M + (size_t)b * ld + d));
  }
  return v;
}

// the new matrix of K clusters from the old one of Kold (average: dsum ->
// dsum2 and dmat; complete: dmat -> dmat2)
template <int LK>
__global__ void __launch_bounds__(32 * FT_Y) k_dense_rebuild(State s, int Kold, int ldold, int K,
                                                              int ld) {
  __shared__ double Mv[32][33];
  long long ti, tj;
  if (!fin_tile(K, ti, tj)) return;
  const int j = (int)tj * 32 + threadIdx.x;
  const bool jin = j < K;
  const int c = jin ? s.dma[j] : 0, d = jin ? s.dmb[j] : -1;
  const double jv = jin ? s.dinv[j] : 0.0;
#pragma unroll
  for (int k0 = 0; k0 < 32; k0 += FT_Y) {
    const int k = k0 + threadIdx.y, i = (int)ti * 32 + k;
    double v = __longlong_as_double((long long)KINF_D);
    if (i < j && jin) {
      const int a = s.dma[i], b = s.dmb[i];
      if (LK == LK_COMPLETE) {
        v = __longlong_as_double((long long)max_new(s.dmat, ldold, a, b, c, d));
      } else {
        const U128 u = sum_new(s.dsum, a, b, c, d, Kold);
        ((ulonglong2 *)s.dsum2)[tri(i, j, K)] = make_ulonglong2(u.lo, u.hi);
        v = entry_mean(u, s.dexp, s.dinv[i], jv);
      }
    }
    Mv[k][threadIdx.x] = v;
  }
  fin_store(LK == LK_COMPLETE ? s.dmat2 : s.dmat, ld, K, ti, tj, Mv);
}

// ---------------------------------------------------------------------------
// the last rounds on the matrix in one launch
// ---------------------------------------------------------------------------
// Below DFIN_K clusters a round is all latency, as in hac_finish.cu: one
// thread-block cluster runs every remaining round (row scans; chain update;
// reciprocal filter and merges; compaction and the new matrix), with the
// hardware cluster barrier between phases.  A terminal whose window holds
// estimates that only the points can decide ends the launch before that
// round changes anything; the host runs the round and comes back.
struct DFinArgs {
  State s;
  NNArgs nn;
  int K, nterm, round, rounds_max, ld;
  const int32_t *order;
  int32_t *order_out, *seg_out;
};

constexpr int DF_T = 1024, DF_W = DF_T / 32;

__device__ __forceinline__ int df_rank() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ int df_count() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void df_sync() {
  __threadfence();
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}

__device__ int df_scan(int v, int *total, int *ws) {  // exclusive, DF_T threads
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
  *total = ws[DF_W - 1];
  __syncthreads();
  return pre + x - v;
}

constexpr int DF_PER = DFIN_K / DF_T;

template <int LK, int F32>
__global__ void __launch_bounds__(DF_T, 1) k_dense_finish(DFinArgs a) {
  __shared__ int s_cid[DFIN_K], s_term[DFIN_K], s_ma[DFIN_K], s_mb[DFIN_K];
  __shared__ double s_inv[DFIN_K];
  __shared__ int ws[DF_W];
  const State &s = a.s;
  const int rank = df_rank(), nct = df_count();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int K = a.K, nterm = a.nterm, round = a.round, ld = a.ld;
  unsigned long long *sum = s.dsum, *sum2 = s.dsum2;
  double *mat = s.dmat, *mat2 = s.dmat2;
  for (int p = threadIdx.x; p < K; p += DF_T) s_cid[p] = a.order[p];
  for (int t = threadIdx.x; t < nterm; t += DF_T) s_term[t] = s.pos[s.term[t]];
  __syncthreads();
  long long searches = 0, naive = 0;
  const int round_end = a.rounds_max > 0 ? round + a.rounds_max : INT_MAX;
  while (K > 1 && round < round_end) {
    for (int t = rank * DF_W + wid; t < nterm; t += nct * DF_W) {
      const int q = s_term[t], ci = s_cid[q];
      const RowNN r = row_scan<F32>(a.nn, mat + (size_t)q * ld, s_cid, K, lane);
      if (lane == 0) {
        s.Ekey[ci] = __longlong_as_double((long long)r.key);
        s.Ecid[ci] = r.kind < 0 ? -1 : r.cid;
        if (r.kind < 0) atomicOr(&s.ctr->err, ERR_NO_NN);
        if (r.kind == 0) atomicAdd(&s.ctr->fin_refused, 1);
      }
    }
    df_sync();
    if (F32 && __ldcg(&s.ctr->fin_refused)) break;  // uniform over the cluster
    searches += nterm;
    naive += (long long)nterm * (K - 1);
    for (int t = rank * DF_T + threadIdx.x; t < nterm; t += nct * DF_T) {
      const int i = s_cid[s_term[t]];
      const int j = __ldcg(&s.Ecid[i]);
      if (j >= 0) s.succ[i] = j;
    }
    df_sync();
    // reciprocal pairs merge, each by one thread (see hac_finish.cu)
    for (int t = rank * DF_T + threadIdx.x; t < nterm; t += nct * DF_T) {
      const int i = s_cid[s_term[t]];
      const int j = __ldcg(&s.Ecid[i]);
      if (j < 0 || __ldcg(&s.succ[j]) != i || !(i < j || __ldcg(&s.isterm[j]) != round)) continue;
      const int lo = min(i, j), hi = max(i, j);
      const int na = __ldcg(&s.csize[lo]), nb = __ldcg(&s.csize[hi]);
      const int r = s.irec[0] + atomicAdd(&s.irecn[0], 1);
      s.m_a[r] = lo;
      s.m_b[r] = hi;
      s.m_h[r] = __ldcg(&s.Ekey[i]);
      s.m_size[r] = na + nb;
      s.m_round[r] = round;
      s.csize[lo] = na + nb;
      s.succ[lo] = -1;
      s.mround[lo] = round;
      s.mround[hi] = round;
      s.alive[hi] = 0;
      s.rootof[hi] = lo;
      s.reloff[hi] = na;
      s.partner[lo] = hi;
    }
    df_sync();
    // chain repair, stable compaction and the old positions of every new
    // cluster, the same in every block
    int c[DF_PER], f[DF_PER], mb[DF_PER], cnt = 0;
#pragma unroll
    for (int r = 0; r < DF_PER; ++r) {
      const int p = threadIdx.x * DF_PER + r;
      c[r] = p < K ? s_cid[p] : -1;
      f[r] = 0;
      mb[r] = -1;
      if (c[r] >= 0 && __ldcg(&s.alive[c[r]])) {
        int sc = __ldcg(&s.succ[c[r]]);
        if (sc >= 0 && __ldcg(&s.mround[sc]) == round) {
          sc = -1;
          if (rank == 0) s.succ[c[r]] = -1;
        }
        if (__ldcg(&s.mround[c[r]]) == round) mb[r] = __ldcg(&s.pos[__ldcg(&s.partner[c[r]])]);
        f[r] = 1 | (sc < 0 ? 1 << 16 : 0);
      }
      cnt += f[r];
    }
    int tot;
    int at = df_scan(cnt, &tot, ws);
    const int K2 = tot & 0xffff;
    if (K2 >= K) {  // no pair merged: cannot happen
      if (rank == 0 && threadIdx.x == 0) atomicOr(&s.ctr->err, ERR_NO_NN);
      break;
    }
#pragma unroll
    for (int r = 0; r < DF_PER; ++r) {
      if (f[r]) {
        const int q = at & 0xffff;
        s_cid[q] = c[r];
        s_ma[q] = threadIdx.x * DF_PER + r;
        s_mb[q] = mb[r];
        s_inv[q] = 1.0 / (double)__ldcg(&s.csize[c[r]]);
        if (f[r] >> 16) {
          s_term[at >> 16] = q;
          if (rank == 0) s.isterm[c[r]] = round + 1;
        }
      }
      at += f[r];
    }
    __syncthreads();
    // positions: read above only for retired cids, which keep their old one
    if (rank == 0)
      for (int p = threadIdx.x; p < K2; p += DF_T) s.pos[s_cid[p]] = p;
    // the new matrix: a warp writes 32 columns of a row of the upper triangle
    const int ld2 = (K2 + 3) & ~3;
    const int segs = (K2 + 31) >> 5;
    for (int t = rank * DF_W + wid; t < K2 * segs; t += nct * DF_W) {
      const int i = t / segs, j = (t - i * segs) * 32 + lane;
      if (j >= K2 || j < i) continue;
      double *out = LK == LK_COMPLETE ? mat2 : mat;
      if (i == j) {
        out[(size_t)i * ld2 + i] = __longlong_as_double((long long)KINF_D);
        continue;
      }
      double v;
      if (LK == LK_COMPLETE) {
        v = __longlong_as_double(
            (long long)max_new(mat, ld, s_ma[i], s_mb[i], s_ma[j], s_mb[j]));
      } else {
        const U128 u = sum_new(sum, s_ma[i], s_mb[i], s_ma[j], s_mb[j], K);
        ((ulonglong2 *)sum2)[tri(i, j, K2)] = make_ulonglong2(u.lo, u.hi);
        v = entry_mean(u, s.dexp, s_inv[i], s_inv[j]);
      }
      out[(size_t)i * ld2 + j] = v;
      out[(size_t)j * ld2 + i] = v;
    }
    if (LK == LK_COMPLETE) {
      double *t = mat;
      mat = mat2;
      mat2 = t;
    } else {
      unsigned long long *t = sum;
      sum = sum2;
      sum2 = t;
    }
    K = K2;
    ld = ld2;
    nterm = tot >> 16;
    ++round;
    df_sync();
  }
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
  if (K > 1 && round > a.round) {  // the lists, segment starts and reciprocals go back
    for (int p = threadIdx.x; p < K; p += DF_T) {
      a.order_out[p] = s_cid[p];
      s.dinv[p] = s_inv[p];
    }
    for (int t = threadIdx.x; t < nterm; t += DF_T) s.term[t] = s_cid[s_term[t]];
    int sz[DF_PER], tot, cnt = 0;
#pragma unroll
    for (int r = 0; r < DF_PER; ++r) {
      const int p = threadIdx.x * DF_PER + r;
      sz[r] = p < K ? __ldcg(&s.csize[s_cid[p]]) : 0;
      cnt += sz[r];
    }
    int at = df_scan(cnt, &tot, ws);
#pragma unroll
    for (int r = 0; r < DF_PER; ++r) {
      const int p = threadIdx.x * DF_PER + r;
      if (p < K) a.seg_out[s_cid[p]] = at;
      at += sz[r];
    }
  }
}

// ---------------------------------------------------------------------------
// FP64 rounds on a packed triangle (hac_run_static)
// ---------------------------------------------------------------------------
// The allocation-free entry point has some MB to spare: once the active
// clusters' packed upper triangle fits (average: the exact 128-bit sum of point
// distances, 16 B per pair, as on the matrix, so that ties are broken alike;
// complete: the distance, 8 B), the FP64 mode fills it from the points over the
// whole GPU and runs every remaining round in one launch.  Without a cache its searches evaluate each big pair again in every
// round, in one warp, and FP64 point pairs are bound by the SM's two-lane FP64
// pipe: 1,024 points of 2-D average took 17.9 ms so, 0.60 here (0.66 with plain FP64 sums in a 6 MiB array).
// Entries are patched in place: a round's survivors add (or take the larger
// of) their partners' entries.
template <int LK>
using TriEntry = typename std::conditional<LK == LK_COMPLETE, double, ulonglong2>::type;

__device__ __forceinline__ double tri_join(double x, double y) { return fmax(x, y); }
__device__ __forceinline__ ulonglong2 tri_join(const ulonglong2 &x, const ulonglong2 &y) {
  U128 s{x.x, x.y};
  u128_add(s, U128{y.x, y.y});
  return make_ulonglong2(s.lo, s.hi);
}

// one warp per pair of clusters
template <int LK, int DP>
__global__ void __launch_bounds__(256) k_tri_fill(State s, const int32_t *order, int K, int cur,
                                                  TriEntry<LK> *tri_) {
  const int lane = threadIdx.x & 31;
  const long long cells = (long long)K * (K - 1) / 2;
  const double *P = s.p64[cur];
  const int32_t *seg = s.seg[cur];
  unsigned long long pp = 0;
  const bool single = K == (int)s.n;  // one thread per pair
  const long long step = (long long)gridDim.x * blockDim.x >> (single ? 0 : 5);
  for (long long t = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> (single ? 0 : 5);
       t < cells; t += step) {
    // column j of the triangle enumerated by columns: t = j (j - 1) / 2 + i
    long long i, j;
    tile_of(t, i, j);
    ++j;
    const int A = order[i], B = order[j];
    int na = single ? 1 : s.csize[A], nb = single ? 1 : s.csize[B], sa = seg[A], sb = seg[B];
    if (nb > na) {
      int x = na;
      na = nb;
      nb = x;
      x = sa;
      sa = sb;
      sb = x;
    }
    double far2 = 0.0;
    U128 acc{0ull, 0ull};
    for (int u = single ? 0 : lane; u < na; u += 32) {
      double x[DP];
#pragma unroll
      for (int k = 0; k < DP; ++k) x[k] = P[(size_t)(sa + u) * DP + k];
      for (int v = 0; v < nb; ++v) {
        double d2 = 0.0;
#pragma unroll
        for (int k = 0; k < DP; ++k) {
          if (k < s.d) {
            const double e = x[k] - P[(size_t)(sb + v) * DP + k];
            d2 = fma(e, e, d2);
          }
        }
        if (LK == LK_COMPLETE)
          far2 = fmax(far2, d2);
        else
          u128_add(acc, fx_of(sqrt(d2), s.dexp));
      }
    }
    if (!single) {
      for (int o = 16; o; o >>= 1) {
        if (LK == LK_COMPLETE)
          far2 = fmax(far2, __shfl_xor_sync(0xffffffffu, far2, o));
        else
          u128_add(acc, u128_shfl_xor(acc, o));
      }
    }
    if (single || lane == 0) {
      if constexpr (LK == LK_COMPLETE)
        tri_[tri(i, j, K)] = sqrt(far2);
      else
        tri_[tri(i, j, K)] = make_ulonglong2(acc.lo, acc.hi);
      pp += (unsigned long long)na * nb;
    }
  }
  for (int o = 16; o; o >>= 1) pp += __shfl_xor_sync(0xffffffffu, pp, o);
  if (lane == 0 && pp) atomicAdd(&s.ctr->point_pairs, pp);
}

struct TriArgs {
  State s;
  int K, nterm, round, rounds_max;  // rounds to run at most (0 = to the end)
  int K0;                           // clusters when the triangle was filled
  int32_t *order;
  void *tri;
};

constexpr int TRI_PER = (TRI_MAX_K + DF_T - 1) / DF_T;

template <int LK>
__global__ void __launch_bounds__(DF_T, 1) k_tri_finish(TriArgs a) {
  // by position in the active list: cid, slot (position when the triangle was
  // filled; the cid's pos, which is not rewritten here); by slot: 1 / size and the
  // partner of this round's merge (-1 none)
  __shared__ int s_cid[TRI_MAX_K], s_slot[TRI_MAX_K], s_term[TRI_MAX_K], s_part[TRI_MAX_K];
  __shared__ double s_inv[TRI_MAX_K];
  __shared__ int ws[DF_W];
  const State &s = a.s;
  const int rank = df_rank(), nct = df_count(), K0 = a.K0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int K = a.K, nterm = a.nterm, round = a.round;
  TriEntry<LK> *T = (TriEntry<LK> *)a.tri;
  for (int p = threadIdx.x; p < K; p += DF_T) {
    const int c = a.order[p], q = s.pos[c];
    s_cid[p] = c;
    s_slot[p] = q;
    s_part[q] = p;  // for the terminals' positions
    s_inv[q] = 1.0 / (double)s.csize[c];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nterm; t += DF_T) s_term[t] = s_part[s.pos[s.term[t]]];
  __syncthreads();
  auto at = [&](int x, int y) -> size_t { return x < y ? tri(x, y, K0) : tri(y, x, K0); };
  long long searches = 0, naive = 0;
  const int round_end = a.rounds_max > 0 ? round + a.rounds_max : INT_MAX;
  while (K > 1 && round < round_end) {
    searches += nterm;
    naive += (long long)nterm * (K - 1);
    for (int t = rank * DF_W + wid; t < nterm; t += nct * DF_W) {
      const int self = s_term[t], q = s_slot[self], ci = s_cid[self];
      const double iq = s_inv[q];
      unsigned long long bk = KINF_D;
      int bp = -1;
#pragma unroll 4
      for (int p = lane; p < K; p += 32) {
        const int r = s_slot[p];
        if (p == self) continue;
        double v;
        if constexpr (LK == LK_COMPLETE) {
          v = __ldcg(T + at(q, r));
        } else {
          const ulonglong2 u = __ldcg(T + at(q, r));
          v = entry_mean(U128{u.x, u.y}, s.dexp, iq, s_inv[r]);
        }
        const unsigned long long k = (unsigned long long)__double_as_longlong(v);
        if ((k < bk || (k == bk && bp >= 0 && s_cid[p] < s_cid[bp]))) {
          bk = k;
          bp = p;
        }
      }
      int bc = bp >= 0 ? s_cid[bp] : INT_MAX;
      warp_argmin_kc(bk, bc);
      if (lane == 0) {
        s.Ekey[ci] = __longlong_as_double((long long)bk);
        s.Ecid[ci] = bc == INT_MAX ? -1 : bc;
        if (bc == INT_MAX) atomicOr(&s.ctr->err, ERR_NO_NN);
      }
    }
    df_sync();
    for (int t = rank * DF_T + threadIdx.x; t < nterm; t += nct * DF_T) {
      const int i = s_cid[s_term[t]];
      const int j = __ldcg(&s.Ecid[i]);
      if (j >= 0) s.succ[i] = j;
    }
    df_sync();
    for (int t = rank * DF_T + threadIdx.x; t < nterm; t += nct * DF_T) {
      const int i = s_cid[s_term[t]];
      const int j = __ldcg(&s.Ecid[i]);
      if (j < 0 || __ldcg(&s.succ[j]) != i || !(i < j || __ldcg(&s.isterm[j]) != round)) continue;
      const int lo = min(i, j), hi = max(i, j);
      const int sz = __ldcg(&s.csize[lo]) + __ldcg(&s.csize[hi]);
      const int r = s.irec[0] + atomicAdd(&s.irecn[0], 1);
      s.m_a[r] = lo;
      s.m_b[r] = hi;
      s.m_h[r] = __ldcg(&s.Ekey[i]);
      s.m_size[r] = sz;
      s.m_round[r] = round;
      s.csize[lo] = sz;
      s.succ[lo] = -1;
      s.mround[lo] = round;
      s.mround[hi] = round;
      s.alive[hi] = 0;
      s.partner[lo] = hi;
    }
    df_sync();
    // chain repair and compaction, the same in every block
    int c[TRI_PER], sl[TRI_PER], f[TRI_PER], cnt = 0;
#pragma unroll
    for (int r = 0; r < TRI_PER; ++r) {
      const int p = threadIdx.x * TRI_PER + r;
      c[r] = p < K ? s_cid[p] : -1;
      sl[r] = p < K ? s_slot[p] : 0;
      f[r] = 0;
      if (c[r] >= 0) {
        int part = -1;
        if (__ldcg(&s.alive[c[r]])) {
          int sc = __ldcg(&s.succ[c[r]]);
          if (sc >= 0 && __ldcg(&s.mround[sc]) == round) {
            sc = -1;
            if (rank == 0) s.succ[c[r]] = -1;
          }
          // a retired cid's pos still is its slot: positions are not rewritten here
          if (__ldcg(&s.mround[c[r]]) == round) part = s.pos[__ldcg(&s.partner[c[r]])];
          f[r] = 1 | (sc < 0 ? 1 << 16 : 0);
        }
        s_part[sl[r]] = part;
      }
      cnt += f[r];
    }
    int tot;
    int pre = df_scan(cnt, &tot, ws);
    const int K2 = tot & 0xffff;
    if (K2 >= K) {  // no pair merged: cannot happen
      if (rank == 0 && threadIdx.x == 0) atomicOr(&s.ctr->err, ERR_NO_NN);
      break;
    }
#pragma unroll
    for (int r = 0; r < TRI_PER; ++r) {
      if (f[r]) {
        const int q = pre & 0xffff;
        s_cid[q] = c[r];
        s_slot[q] = sl[r];
        s_inv[sl[r]] = 1.0 / (double)__ldcg(&s.csize[c[r]]);
        if (f[r] >> 16) {
          s_term[pre >> 16] = q;
          if (rank == 0) s.isterm[c[r]] = round + 1;
        }
      }
      pre += f[r];
    }
    __syncthreads();
    // entries of the survivors: a warp per merged cluster and 32 others
    const int segs = (K2 + 31) >> 5;
    for (int t = rank * DF_W + wid; t < K2 * segs; t += nct * DF_W) {
      const int x = s_slot[t / segs], b = s_part[x];
      if (b < 0) continue;  // did not merge (uniform over the warp)
      const int p = (t % segs) * 32 + lane;
      if (p >= K2) continue;
      const int y = s_slot[p], d = s_part[y];
      if (y == x || (d >= 0 && y < x)) continue;  // both merged: the lower slot's warp does it
      TriEntry<LK> v = tri_join(__ldcg(T + at(x, y)), __ldcg(T + at(b, y)));
      if (d >= 0) v = tri_join(v, tri_join(__ldcg(T + at(x, d)), __ldcg(T + at(b, d))));
      T[at(x, y)] = v;
    }
    K = K2;
    nterm = tot >> 16;
    ++round;
    df_sync();
  }
  if (rank != 0) return;
  if (K > 1) {  // stopped by the round limit: the lists go back
    for (int p = threadIdx.x; p < K; p += DF_T) a.order[p] = s_cid[p];
    for (int t = threadIdx.x; t < nterm; t += DF_T) s.term[t] = s_cid[s_term[t]];
  }
  if (threadIdx.x != 0) return;
  s.ctr->nactive = K;
  s.ctr->nterm = nterm;
  s.ctr->nmerges += a.K - K;
  s.ctr->ltests += (unsigned long long)naive;
  s.ctr->fin_rounds = round - a.round;
  s.ctr->fin_searches = searches;
  s.ctr->fin_naive = naive;
  s.idone[0] = K <= 1;
  s.iact[0] = K;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <typename F>
void launch_2d_tiles(F kernel, long long tiles, int threads_x, cudaStream_t st,
                     const SweepArgs &a) {
  const unsigned gx = (unsigned)std::min<long long>(tiles, 65535);
  const unsigned gy = (unsigned)((tiles + gx - 1) / gx);
  kernel<<<dim3(gx, gy), threads_x, 0, st>>>(a);
}

int sweep(hac_ctx *h, cudaStream_t st, const SweepArgs &a) {
  const State &s = h->s;
  const bool f32 = s.prec == HAC_PREC_F32_RECHECK;
  // rows per thread: 4 (2 for 16-wide FP32 rows and for FP64), for 2-3
  // resident tiles per SM
  const int ppt = f32 && s.dp <= 8 ? HAC_DS_PPT8 : 2;
  const long long TI = (long long)DS_TPB * ppt;
  SweepArgs b = a;
  b.nb = (a.N + TI - 1) / TI;
  const long long tiles = b.nb * (b.nb + 1) / 2;
  if (f32) {
    constexpr int P8 = HAC_DS_PPT8;
    switch (s.d) {  // specialised on the true dimension
      case 1: launch_2d_tiles(k_dense_sweep32<1, 2, P8>, tiles, DS_TPB, st, b); break;
      case 2: launch_2d_tiles(k_dense_sweep32<2, 2, P8>, tiles, DS_TPB, st, b); break;
      case 3: launch_2d_tiles(k_dense_sweep32<3, 4, P8>, tiles, DS_TPB, st, b); break;
      case 4: launch_2d_tiles(k_dense_sweep32<4, 4, P8>, tiles, DS_TPB, st, b); break;
      case 5: launch_2d_tiles(k_dense_sweep32<5, 8, P8>, tiles, DS_TPB, st, b); break;
      case 6: launch_2d_tiles(k_dense_sweep32<6, 8, P8>, tiles, DS_TPB, st, b); break;
      case 7: launch_2d_tiles(k_dense_sweep32<7, 8, P8>, tiles, DS_TPB, st, b); break;
      case 8: launch_2d_tiles(k_dense_sweep32<8, 8, P8>, tiles, DS_TPB, st, b); break;
      case 9: launch_2d_tiles(k_dense_sweep32<9, 16, 2>, tiles, DS_TPB, st, b); break;
      case 10: launch_2d_tiles(k_dense_sweep32<10, 16, 2>, tiles, DS_TPB, st, b); break;
      case 11: launch_2d_tiles(k_dense_sweep32<11, 16, 2>, tiles, DS_TPB, st, b); break;
      case 12: launch_2d_tiles(k_dense_sweep32<12, 16, 2>, tiles, DS_TPB, st, b); break;
      case 13: launch_2d_tiles(k_dense_sweep32<13, 16, 2>, tiles, DS_TPB, st, b); break;
      case 14: launch_2d_tiles(k_dense_sweep32<14, 16, 2>, tiles, DS_TPB, st, b); break;
      case 15: launch_2d_tiles(k_dense_sweep32<15, 16, 2>, tiles, DS_TPB, st, b); break;
      default: launch_2d_tiles(k_dense_sweep32<16, 16, 2>, tiles, DS_TPB, st, b);
    }
  } else {
    switch (s.d) {
      case 1: launch_2d_tiles(k_dense_sweep64<1, 2, 2>, tiles, DS_TPB, st, b); break;
      case 2: launch_2d_tiles(k_dense_sweep64<2, 2, 2>, tiles, DS_TPB, st, b); break;
      case 3: launch_2d_tiles(k_dense_sweep64<3, 4, 2>, tiles, DS_TPB, st, b); break;
      case 4: launch_2d_tiles(k_dense_sweep64<4, 4, 2>, tiles, DS_TPB, st, b); break;
      case 5: launch_2d_tiles(k_dense_sweep64<5, 8, 2>, tiles, DS_TPB, st, b); break;
      case 6: launch_2d_tiles(k_dense_sweep64<6, 8, 2>, tiles, DS_TPB, st, b); break;
      case 7: launch_2d_tiles(k_dense_sweep64<7, 8, 2>, tiles, DS_TPB, st, b); break;
      case 8: launch_2d_tiles(k_dense_sweep64<8, 8, 2>, tiles, DS_TPB, st, b); break;
      case 9: launch_2d_tiles(k_dense_sweep64<9, 16, 2>, tiles, DS_TPB, st, b); break;
      case 10: launch_2d_tiles(k_dense_sweep64<10, 16, 2>, tiles, DS_TPB, st, b); break;
      case 11: launch_2d_tiles(k_dense_sweep64<11, 16, 2>, tiles, DS_TPB, st, b); break;
      case 12: launch_2d_tiles(k_dense_sweep64<12, 16, 2>, tiles, DS_TPB, st, b); break;
      case 13: launch_2d_tiles(k_dense_sweep64<13, 16, 2>, tiles, DS_TPB, st, b); break;
      case 14: launch_2d_tiles(k_dense_sweep64<14, 16, 2>, tiles, DS_TPB, st, b); break;
      case 15: launch_2d_tiles(k_dense_sweep64<15, 16, 2>, tiles, DS_TPB, st, b); break;
      default: launch_2d_tiles(k_dense_sweep64<16, 16, 2>, tiles, DS_TPB, st, b);
    }
  }
  CK(cudaGetLastError());
  return HAC_OK;
}

// grid of the 32 x 32 tiles of the upper triangle of a K x K matrix
dim3 tile_grid(int K) {
  const long long nt = (K + 31) / 32, tiles = nt * (nt + 1) / 2;
  const unsigned gx = (unsigned)std::min<long long>(tiles, 65535);
  return dim3(gx, (unsigned)((tiles + gx - 1) / gx));
}
const dim3 kTileBlock(32, FT_Y);

int64_t dense_threshold(const hac_ctx *h) {
  return h->dense_k >= 0 ? h->dense_k : h->dense_def;
}

int dense_ld(int64_t K) { return (int)((K + 3) & ~(int64_t)3); }

template <int LK, int F32>
void launch_single(hac_ctx *h, cudaStream_t st, int K, float scl, int es, float inv_scl) {
  const State &s = h->s;
  const float *p32 = s.p32[h->pcur];
  const double *p64 = s.p64[h->pcur];
  const dim3 g = tile_grid(K);
  switch (s.dp) {
    case 2: k_dense_single<LK, 2, F32><<<g, kTileBlock, 0, st>>>(s, p32, p64, K, scl, es, inv_scl); break;
    case 4: k_dense_single<LK, 4, F32><<<g, kTileBlock, 0, st>>>(s, p32, p64, K, scl, es, inv_scl); break;
    case 8: k_dense_single<LK, 8, F32><<<g, kTileBlock, 0, st>>>(s, p32, p64, K, scl, es, inv_scl); break;
    default: k_dense_single<LK, 16, F32><<<g, kTileBlock, 0, st>>>(s, p32, p64, K, scl, es, inv_scl);
  }
}

template <int LK>
void launch_rq(const State &s, const int32_t *order, int m, int cur, cudaStream_t st) {
  const int g = device_sms() * 4;
  switch (s.dp) {
    case 2: k_drq_eval<LK, 2><<<g, RQ_TPB, 0, st>>>(s, order, m, cur); break;
    case 4: k_drq_eval<LK, 4><<<g, RQ_TPB, 0, st>>>(s, order, m, cur); break;
    case 8: k_drq_eval<LK, 8><<<g, RQ_TPB, 0, st>>>(s, order, m, cur); break;
    default: k_drq_eval<LK, 16><<<g, RQ_TPB, 0, st>>>(s, order, m, cur);
  }
  k_drq_fin<LK><<<grid_for(m, TPB), TPB, 0, st>>>(s, m);
}

// FP64 re-score of the first m listed pairs (they then hold exact values)
int recheck(hac_ctx *h, cudaStream_t st, int m) {
  State &s = h->s;
  if (m <= 0) return HAC_OK;
  int rc = relayout_if_stale(h, st);
  if (rc) return rc;
  const int32_t *order = s.order[h->ocur];
  CK(cudaMemsetAsync(s.drq_acc, 0, (size_t)m * LIMBS * sizeof(unsigned long long), st));
  k_drq_count<<<grid_for(m, TPB), TPB, 0, st>>>(s, order, m);
  k_drq_scan<<<1, 1024, 0, st>>>(s, m);
  if (s.linkage == LK_COMPLETE)
    launch_rq<LK_COMPLETE>(s, order, m, h->pcur, st);
  else
    launch_rq<LK_AVERAGE>(s, order, m, h->pcur, st);
  h->launches += 4;
  CK(cudaGetLastError());
  return HAC_OK;
}

// Arguments of the row scans in the current state
void nn_args(const hac_ctx *h, int K, NNArgs &a, bool *intb) {
  const State &s = h->s;
  a = NNArgs{};
  a.dmat = s.dmat;
  a.ld = s.dld;
  a.K = K;
  a.order = s.order[h->ocur];
  a.pos = s.pos;
  a.list = s.term;
  a.delta = (double)s.delta_pts;
  // average: FP32 partial sums of at most 32 terms on top of a distance's bound
  a.rho = ((double)s.d + (s.linkage == LK_COMPLETE ? 16.0 : 48.0)) * 5.9604644775390625e-8;
  a.Ekey = s.Ekey;
  a.Ecid = s.Ecid;
  a.drq_a = s.drq_a;
  a.drq_b = s.drq_b;
  a.drq_cap = s.drq_cap;
  a.ctr = s.ctr;
  // absolute term: a truncation below one unit 2^dexp on each side (the FP32
  // partial sums and the FP64 re-score's distances) and the flush of scaled
  // squared distances below 2^-126 (distances below 2^(-63-dsk))
  a.eta = (std::ldexp(1.0, -63 - s.dsk) +
           (s.linkage == LK_COMPLETE ? 0.0 : 2.0 * std::ldexp(1.0, s.dexp))) * (1.0 + 1e-9);
  const bool f32 = s.prec == HAC_PREC_F32_RECHECK;
  // integer bounds when the estimates carry no relative-to-scale absolute
  // term and the lone estimate's bound is within the 4e-6 the height
  // convention allows; above m0 = 2^30 eta the absolute term is within
  // 2^-30 of an entry and joins rho
  const double rho_i = a.rho + std::ldexp(1.0, -30);
  *intb = f32 && a.delta == 0.0 && rho_i <= 4e-6;
  a.nu = (unsigned long long)std::ceil(std::ldexp(rho_i / (1.0 - rho_i), 53) * (1.0 + 1e-6)) + 2;
  a.nl = 2 * ((unsigned long long)std::ceil(std::ldexp(rho_i, 53) * (1.0 + 1e-6)) + 2);
  const double m0 = std::ldexp(a.eta, 30);
  memcpy(&a.m0, &m0, 8);
  const double m0up = 2.0 * m0;
  memcpy(&a.m0up, &m0up, 8);
}

// Buffers, sized once per handle for the largest matrix it can need: three
// (average: two for the sums, one for the means; the first two together hold
// the sweep's limbs) or two (complete) of 8 B per entry.  HAC_ENOMEM if the
// matrices do not fit (the instance then stays on the range-query search).
int dense_alloc(hac_ctx *h, int64_t cap) {
  State &s = h->s;
  const int rqcap = (int)std::min<int64_t>(std::max<int64_t>(4 * cap, 1 << 16), 1 << 22);
  const size_t buf = (size_t)dense_ld(cap) * cap;  // doubles
  const int nbuf = s.linkage == LK_COMPLETE ? 2 : 3;
  int rc = dalloc(h, &h->dense_buf, nbuf * buf);
  if (rc) return rc;
  SlabAlloc m;
  m.add(&s.dma, cap);
  m.add(&s.dmb, cap);
  m.add(&s.dinv, cap);
  m.add(&s.drq_a, rqcap);
  m.add(&s.drq_b, rqcap);
  m.add(&s.drq_pre, rqcap + 1);
  m.add(&s.drq_acc, LIMBS * (size_t)rqcap);
  m.add(&s.dpend[0], cap);
  m.add(&s.dpend[1], cap);
  if ((rc = m.commit(h))) return rc;
  s.drq_cap = rqcap;
  h->dense_cap = cap;
  h->dense_stride = buf;
  return HAC_OK;
}

}  // namespace

// Default largest matrix of a run.  Each line lies where the whole run took as
// long on either side (ms, FP32 mode, 128 cache slots, mixture data):
// average: the range-query rounds prune well in low dimension and poorly above
// 8.  A run of few points starts on the matrix (d = 5, 8,000 points: 4.65, at
// 4,096 clusters 5.27; 10,000: 5.88 / 5.72); above, a later switch is better
// while clusters are few points each (the sweep then flushes every column), a
// larger matrix again once the tree's big pairs weigh more:
//   d = 2, 100,000 points: 10.4 at 4,096, 11.2 at 8,192; 10^6: 170 / 168
//   d = 5, 20,001 points: 11.0 at 4,096, 11.8 at 8,192, 20.4 at 16,384;
//     200,000: 64.8 at 4,096, 49.7 at 8,192; 10^6: 463 / 440 / 426 at 16,384
//   d = 10, 20,001 points: 19.5 from the start, 28.8 at 8,192; 30,001: 37.9
//     from the start, 42.7 at 16,384; 100,000: 191 at 16,384, 189 at 20,000,
//     190 at 32,768 (and 16 GB less to allocate); 16-D lattice, 10^6 points:
//     11.5 s at 32,768, 8.3 s at 65,536
// complete (from the start or not at all): FP32 d = 2, 20,001 points 8.6
// against 13.1 on the range query, 30,001: 15.5 / 14.2; d = 5, 30,001: 19.6 /
// 22.0, 32,768: 23.8 / 22.9; FP64, whose point pairs cost 60 times as much,
// 35 / 110 at 30,001 points in 5-D.
// The matrices (24 or 16 B per entry) take at most half of the device memory
// free at the start of the run.
int64_t dense_default(int64_t n, int d, int linkage, int prec) {
  int64_t k;
  if (linkage == LK_COMPLETE)
    k = prec == HAC_PREC_F64 || d > 8 ? 32768 : d <= 3 ? 24576 : 30000;
  else if (d > 8)
    k = n <= 32768 ? 32768 : std::min<int64_t>(65536, std::max<int64_t>(20000, n / 16));
  else if (n <= 8192)
    k = 8192;
  else if (d <= 3)
    k = n <= 250000 ? 4096 : 8192;
  else
    k = std::min<int64_t>(16384, std::max<int64_t>(4096, n / 16));
  const double per = linkage == LK_COMPLETE ? 16.0 : 24.0;
  size_t fr = 0, tot = 0;
  if (cudaMemGetInfo(&fr, &tot) == cudaSuccess)
    k = std::min<int64_t>(k, (int64_t)std::sqrt(0.5 * (double)fr / per));
  else
    cudaGetLastError();
  return k;
}

// unit of the fixed-point sums: (n/2)^2 x the largest point distance < 2^126 units
void set_sum_unit(hac_ctx *h) {
  State &s = h->s;
  const double dmax = 2.0 * (double)s.coord_scale * std::sqrt((double)s.d) * (1.0 + 1e-5);
  const double smax = 0.25 * (double)h->lay_n * (double)h->lay_n * dmax;
  s.dexp = smax > 0.0 ? (int)std::floor(std::log2(smax)) + 1 - 126 : -1000;
}

// Complete linkage keeps the whole matrix only from the first round on (at
// most the threshold's points); average linkage switches in mid-run too.
bool dense_allowed(const hac_ctx *h, int K) {
  const State &s = h->s;
  if (closed_form(s.linkage) || s.max_inst != 1 || s.noprune || K < 2) return false;
  if ((int64_t)K > dense_threshold(h)) return false;
  return s.linkage == LK_AVERAGE || K == h->n;
}

int dense_reserve(hac_ctx *h, int K) {
  if (!dense_allowed(h, K)) return 0;
  if (h->dense_cap >= K) return 1;
  const int rc = dense_alloc(h, std::min<int64_t>(dense_threshold(h), h->n));
  if (rc == HAC_OK) return 1;
  h->dense_k = 0;  // no room: the instance stays on the range-query search
  return 0;
}

int dense_maybe_enter(hac_ctx *h, cudaStream_t st, int K, RoundCtl &ctl) {
  State &s = h->s;
  if (s.dense) return 1;
  if (!dense_reserve(h, K)) return 0;
  s.dk = K;
  s.dld = dense_ld(K);
  set_sum_unit(h);
  // the FP32 copy scaled by 2^k toward |coordinate| <= 2^40 (squared
  // distances stay below 2^86 for d <= 16; k >= 0 keeps the scaling exact)
  int k = 0;
  if (s.p32_max > 0.0)
    k = std::max(0, std::min(100, 40 - (int)std::ceil(std::log2(s.p32_max))));
  s.dsk = k;
  const float scl = std::ldexp(1.0f, k);
  const int es = s.dexp + k;
  const bool f32 = s.prec == HAC_PREC_F32_RECHECK;
  const bool single = (int64_t)K == h->lay_n;
  double *b0 = h->dense_buf, *b1 = b0 + h->dense_stride, *b2 = b1 + h->dense_stride;
  k_dense_init<<<grid_for(K, TPB), TPB, 0, st>>>(
      s, s.order[h->ocur], K, single ? (unsigned long long)K * (K - 1) / 2 : 0ull);
  if (single) {
    if (ctl.eb0) cudaEventRecord(ctl.eb0, st);
    const float inv_scl = std::ldexp(1.0f, -k);
    if (s.linkage == LK_COMPLETE) {
      s.dmat = b0;
      s.dmat2 = b1;
      if (f32)
        launch_single<LK_COMPLETE, 1>(h, st, K, scl, es, inv_scl);
      else
        launch_single<LK_COMPLETE, 0>(h, st, K, scl, es, inv_scl);
    } else {
      s.dsum = (unsigned long long *)b0;
      s.dsum2 = (unsigned long long *)b1;
      s.dmat = b2;
      if (f32)
        launch_single<LK_AVERAGE, 1>(h, st, K, scl, es, inv_scl);
      else
        launch_single<LK_AVERAGE, 0>(h, st, K, scl, es, inv_scl);
    }
    CK(cudaGetLastError());
    if (ctl.eb1) cudaEventRecord(ctl.eb1, st);
  } else {
    const size_t cells = (size_t)K * (K - 1) / 2;
    CK(cudaMemsetAsync(b0, 0, cells * LIMBS * sizeof(unsigned long long), st));
    SweepArgs a{};
    a.p32 = s.p32[h->pcur];
    a.p64 = s.p64[h->pcur];
    a.plab = s.plab[h->pcur];
    a.pos = s.pos;
    a.N = h->lay_n;
    a.dk = K;
    a.e = s.dexp;
    a.scl = scl;
    a.es = es;
    a.sum = (unsigned long long *)b0;
    a.ctr = s.ctr;
    if (ctl.eb0) cudaEventRecord(ctl.eb0, st);
    int rc = sweep(h, st, a);
    if (rc) return rc;
    if (ctl.eb1) cudaEventRecord(ctl.eb1, st);
    k_dense_pack<<<grid_for((int64_t)cells, TPB), TPB, 0, st>>>(
        (const unsigned long long *)b0, (unsigned long long *)b2, cells, f32);
    s.dsum = (unsigned long long *)b2;
    s.dsum2 = (unsigned long long *)b1;
    s.dmat = b0;
    k_dense_mean<<<tile_grid(K), kTileBlock, 0, st>>>(s, K);
    CK(cudaGetLastError());
    h->launches += 2;
    ctl.dense_launches += 2;
  }
  if (ctl.eb0) {
    CK(cudaEventSynchronize(ctl.eb1));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, ctl.eb0, ctl.eb1);
    ctl.ms_dense += ms;
  }
  h->launches += 2;
  ctl.dense_launches += 2;
  s.dense = 1;
  h->dense_k0 = K;
  return 1;
}

int dense_search(hac_ctx *h, cudaStream_t st, int K, int nterm, RoundCtl &ctl) {
  State &s = h->s;
  NNArgs a;
  bool intb;
  nn_args(h, K, a, &intb);
  a.nlist = nterm;
  const bool f32 = s.prec == HAC_PREC_F32_RECHECK;
  // every pass settles the listed estimates, at most drq_cap of them
  const long long passes = 64 + (long long)K * K / std::max(1, s.drq_cap);
  for (long long it = 0;; ++it) {
    if (it >= passes) return HAC_EINTERNAL;
    CK(cudaMemsetAsync(&s.ctr->npend, 0, sizeof(int32_t), st));
    CK(cudaMemsetAsync(&s.ctr->nrq, 0, sizeof(int32_t), st));
    a.pend_out = s.dpend[it & 1];
    const int blocks = std::max(1, std::min(cdiv(a.nlist, 8), device_sms() * 16));
    if (intb)
      k_dense_nn<2><<<blocks, 256, 0, st>>>(a);
    else if (f32)
      k_dense_nn<1><<<blocks, 256, 0, st>>>(a);
    else
      k_dense_nn<0><<<blocks, 256, 0, st>>>(a);
    CK(cudaGetLastError());
    h->launches += 1;
    ctl.searches += a.nlist;
    if (!f32) break;
    int cnt[2];  // npend, nrq are not adjacent: two reads
    CK(cudaMemcpyAsync(&cnt[0], &s.ctr->npend, sizeof(int), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(&cnt[1], &s.ctr->nrq, sizeof(int), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (cnt[0] == 0) break;
    const int m = std::min(cnt[1], s.drq_cap);
    ctl.dense_launches += 4;
    int rc = recheck(h, st, m);
    if (rc) return rc;
    ctl.dense_rechecks += m;
    a.list = s.dpend[it & 1];
    a.nlist = cnt[0];
  }
  return HAC_OK;
}

// after the compaction: the matrix of the K clusters left, from Kold's
int dense_update(hac_ctx *h, cudaStream_t st, int round, int Kold, int K) {
  State &s = h->s;
  if (K < 2) return HAC_OK;
  const int ld = dense_ld(K);
  k_dense_map<<<grid_for(Kold, TPB), TPB, 0, st>>>(s, s.order[h->ocur ^ 1], Kold, round);
  if (s.linkage == LK_COMPLETE) {
    k_dense_rebuild<LK_COMPLETE><<<tile_grid(K), kTileBlock, 0, st>>>(s, Kold, s.dld, K, ld);
    std::swap(s.dmat, s.dmat2);
  } else {
    k_dense_rebuild<LK_AVERAGE><<<tile_grid(K), kTileBlock, 0, st>>>(s, Kold, s.dld, K, ld);
    std::swap(s.dsum, s.dsum2);
  }
  s.dk = K;
  s.dld = ld;
  h->launches += 2;
  CK(cudaGetLastError());
  return HAC_OK;
}

int dense_finish(hac_ctx *h, cudaStream_t st, int K, int nterm, int round, int64_t limit,
                 Counters *c) {
  State &s = h->s;
  DFinArgs a{};
  bool intb;
  nn_args(h, K, a.nn, &intb);
  a.s = s;
  a.K = K;
  a.nterm = nterm;
  a.round = round;
  a.rounds_max = (int)std::min<int64_t>(limit, INT32_MAX / 2);
  a.ld = s.dld;
  a.order = s.order[h->ocur];
  a.order_out = s.order[h->ocur];
  a.seg_out = s.seg[h->pcur ^ 1];
  const bool f32 = s.prec == HAC_PREC_F32_RECHECK;
  const bool comp = s.linkage == LK_COMPLETE;
  auto kern = comp ? (!f32 ? k_dense_finish<LK_COMPLETE, 0>
                           : intb ? k_dense_finish<LK_COMPLETE, 2> : k_dense_finish<LK_COMPLETE, 1>)
                   : (!f32 ? k_dense_finish<LK_AVERAGE, 0>
                           : intb ? k_dense_finish<LK_AVERAGE, 2> : k_dense_finish<LK_AVERAGE, 1>);
  CK(cudaMemsetAsync(&s.ctr->fin_refused, 0, sizeof(int32_t), st));
  // (whole 3-D runs, ms, with 1 / 4 / 8 / 16 blocks: average 64 clusters 0.277 / 0.269 /
  // 0.270 / 0.271, 200 0.413 / 0.351 / 0.341 / 0.333, 800 1.62 / 0.75 / 0.61 / 0.53)
  const int nct = K <= 64 ? 1 : K <= 200 ? 8 : 16;
  int rc = launch_cluster((const void *)kern, nct, DF_T, 0, &a, st);
  if (rc) return rc;
  h->launches += 1;
  CK(cudaMemcpyAsync(c, s.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  if (c->fin_rounds > 0) {
    h->lay_stale = 1;
    if (c->fin_rounds & 1) {
      if (comp)
        std::swap(s.dmat, s.dmat2);
      else
        std::swap(s.dsum, s.dsum2);
    }
    s.dk = c->nactive;
    s.dld = dense_ld(c->nactive);
  }
  return HAC_OK;
}

size_t tri_bytes(int linkage) {
  return linkage == LK_COMPLETE ? sizeof(TriEntry<LK_COMPLETE>) : sizeof(TriEntry<LK_AVERAGE>);
}

// The remaining rounds (at most `limit` of them, 0 = all) of an FP64 run on the
// packed triangle at h->tri (room for h->tri_cap clusters), which the first call
// fills; the counters come back in *c.
int tri_finish(hac_ctx *h, cudaStream_t st, int K, int nterm, int round, int64_t limit,
               Counters *c) {
  State &s = h->s;
  int32_t *order = s.order[h->ocur];
  const int g = device_sms() * 8;
  const bool comp = s.linkage == LK_COMPLETE;
#define TRI_FILL(DP)                                                                      \
  (comp ? k_tri_fill<LK_COMPLETE, DP><<<g, 256, 0, st>>>(                                 \
              s, order, K, h->pcur, (TriEntry<LK_COMPLETE> *)h->tri)                      \
        : k_tri_fill<LK_AVERAGE, DP><<<g, 256, 0, st>>>(                                  \
              s, order, K, h->pcur, (TriEntry<LK_AVERAGE> *)h->tri))
  if (!h->tri_k0) {
    h->tri_k0 = K;
    set_sum_unit(h);
    switch (s.dp) {
      case 2: TRI_FILL(2); break;
      case 4: TRI_FILL(4); break;
      case 8: TRI_FILL(8); break;
      default: TRI_FILL(16);
    }
    CK(cudaGetLastError());
    h->launches += 1;
  }
#undef TRI_FILL
  TriArgs a{};
  a.s = s;
  a.K = K;
  a.nterm = nterm;
  a.round = round;
  a.rounds_max = (int)std::min<int64_t>(limit, INT32_MAX / 2);
  a.K0 = h->tri_k0;
  a.order = order;
  a.tri = h->tri;
  // (static calls in 3-D, ms, with 1 / 4 / 8 / 16 blocks: average 64 clusters 0.266 / 0.263
  // / 0.266 / 0.266, 200 0.410 / 0.333 / 0.327 / 0.316, 800 1.89 / 0.87 / 0.70 / 0.61)
  const int nct = K <= 64 ? 1 : K <= 200 ? 8 : 16;
  int rc = launch_cluster(comp ? (const void *)k_tri_finish<LK_COMPLETE>
                               : (const void *)k_tri_finish<LK_AVERAGE>,
                          nct, DF_T, 0, &a, st);
  if (rc) return rc;
  h->launches += 1;
  CK(cudaMemcpyAsync(c, s.ctr, sizeof(Counters), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  return HAC_OK;
}

}  // namespace hacg
