// Host and device internals shared by the library's translation units
// (core rounds, big-pair evaluation, serving); not part of the C ABI.
#pragma once

#include "hac.h"
#include "hac_internal.cuh"
#include "hac_dev.cuh"

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <new>
#include <vector>

namespace hacg {

constexpr int TPB = 256;

__host__ __device__ inline int cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

// Bounds, summaries and screening square coordinates in FP32, so the clustering
// runs at a scale that FP32 holds: an input whose largest recentred coordinate is
// outside [FIN_SCALE_LO, FIN_SCALE_HI) is multiplied by 2^-unit_exp, which takes
// it to [0.5, 1), and heights are multiplied back as they leave (both exact,
// unless a height itself is outside FP64's normal range).  Unscaled, coordinates
// from 2^63 on had infinite lower bounds and lost their nearest neighbours, and
// below 2^-50 every FP32 variance was the least subnormal.
__host__ __device__ inline int unit_exp(double scale) {
  if (!(scale > 0.0) || (scale >= FIN_SCALE_LO && scale < FIN_SCALE_HI)) return 0;
  int e;
  frexp(scale, &e);
  return e < -1023 ? -1023 : e > 1023 ? 1023 : e;
}
// the middle of [lo, hi] (halved first: the sum may be beyond FP64)
__host__ __device__ inline double box_centre(double lo, double hi) { return 0.5 * lo + 0.5 * hi; }
// a height in input units (avg-2: squared units)
__host__ __device__ inline double unit_height(double h, double unit, bool squared) {
  h *= unit;
  return squared ? h * unit : h;
}

// ---------------------------------------------------------------------------
// pair-distance cache slots (Section 5): the write protocol
// ---------------------------------------------------------------------------
constexpr unsigned long long CKEY_BUSY = ~1ull;  // a slot whose value is being written

__device__ __forceinline__ unsigned long long slot_key(const State &s, size_t idx) {
  return *(volatile unsigned long long *)&s.ckey[idx];
}

// an empty slot, or one whose neighbour has merged since (stale generation)
__device__ __forceinline__ bool slot_free(const State &s, unsigned long long cur) {
  if (cur == CKEY_EMPTY) return true;
  if (cur == CKEY_BUSY) return false;
  return (unsigned)cur != (unsigned)s.gen[(int)(cur >> 32)];
}

// Claim slot idx (holding `cur`) by CAS to BUSY, write the value, then
// publish the key: concurrent writers skip BUSY slots, so a slot's key and
// value always come from the same writer.  Readers run in later kernels.
__device__ inline bool slot_put(const State &s, size_t idx, unsigned long long cur,
                         unsigned long long want, double v, float e, int part = 0) {
  if (atomicCAS(&s.ckey[idx], cur, CKEY_BUSY) != cur) return false;
  s.cval[idx] = v;
  s.cerr[idx] = e;
  s.cpart[idx] = part;
  __threadfence();
  atomicExch(&s.ckey[idx], want);
  return true;
}

// Insert (nbr -> v, e) into the table of `owner` if there is a free slot;
// an entry already present is kept (a partial one is completed by it).
__device__ inline void cache_insert(const State &s, int owner, int nbr, int nbr_gen, double v, float e) {
  const int S = s.cache_slots;
  const unsigned long long want = ckey_of(nbr, nbr_gen);
  const size_t base = (size_t)owner * S;
  int t = (int)(((unsigned)nbr * 2654435761u) % (unsigned)S);
  for (int q = 0; q < S; ++q, t = t + 1 == S ? 0 : t + 1) {
    // a free slot only turns BUSY or live within a kernel, so this ends
    for (;;) {
      const unsigned long long cur = slot_key(s, base + t);
      if (cur == want) {
        if (s.cpart[base + t] != 0) slot_put(s, base + t, cur, want, v, e);
        return;
      }
      if (!slot_free(s, cur)) break;
      if (slot_put(s, base + t, cur, want, v, e)) {
        s.cused[owner] = 1;
        return;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// big pairs: sizes of the GPU-wide evaluation
// ---------------------------------------------------------------------------
constexpr int BIG_TPB = 256;       // threads per tile
constexpr int BIG_TILE = BIG_TPB * 2;  // narrowest tile along the larger cluster
constexpr int BIG_MAXT = 32768; // tiles per request at most (chunks widen to fit)
constexpr int BIG_BATCH = 1024;    // requests per batch (one scan block of 32 warps)

// Three kinds of request, each its own tile list and kernel:
//   0  FP32, larger cluster >= 256 x 8 points: 8 of its points per thread
//      (4 for d > 8)
//   1  FP32, smaller requests: 2 points per thread
//   2  FP64 (exact values wanted): 2 points per thread
// A tile is (points of the larger cluster) x (a chunk of the smaller one).
constexpr int BK_KINDS = 3;
__host__ __device__ inline int bk_ppt(int kind, int d) { return kind == 0 ? (d <= 8 ? 8 : 4) : 2; }
__host__ __device__ inline int bk_width(int kind, int d) { return BIG_TPB * bk_ppt(kind, d); }

__host__ __device__ inline int bk_kind(int nL, bool exact, int d) {
  return exact ? 2 : nL >= bk_width(0, d) ? 0 : 1;
}

// chunk of the smaller cluster per tile (2048 points FP32, 1024 FP64),
// widened so that a request has at most max(BIG_MAXT, tiles along the larger
// cluster) tiles
__host__ __device__ inline int bk_chunk(int kind, int nL, int nS, int d) {
  const int w = bk_width(kind, d);
  const int tl = (nL + w - 1) / w;
  int c = kind == 2 ? 1024 : 2048;
  const int maxts = BIG_MAXT / tl > 1 ? BIG_MAXT / tl : 1;
  if ((nS + c - 1) / c > maxts) c = (nS + maxts - 1) / maxts;
  return c;
}

// Schedule of one batch, in s.bsched (ints):
//   [0, B)            tile start of each request in bpart (all kinds)
//   [B, 2B)           tile count of each request
//   per kind k at 2B + k (2B + 1): B request indices, then B + 1 tile prefix
//   at 2B + 3 (2B + 1): n_k (requests of kind k), T_k (tiles), next_k (work
//   counter) for each kind
constexpr int BS_B = BIG_BATCH;
constexpr int BS_LIST = 2 * BS_B;
constexpr int BS_META = 2 * BS_B + BK_KINDS * (2 * BS_B + 1);
constexpr int BS_SIZE = BS_META + 3 * BK_KINDS;

}  // namespace hacg

// ---------------------------------------------------------------------------
// instance
// ---------------------------------------------------------------------------
struct hac_ctx {
  hacg::State s{};
  int64_t n = 0;
  int d = 0;
  hac_dtype dt = HAC_F64;
  hac_linkage lk = HAC_WARD;
  void *raw = nullptr;          // device copy of the input points (input order)
  cudaStream_t own = nullptr;
  std::vector<void *> allocs;
  int64_t bytes = 0;
  // sort scratch
  uint64_t *keys[2] = {nullptr, nullptr};
  int32_t *vals[2] = {nullptr, nullptr};
  int32_t *hist = nullptr, *hbs = nullptr;
  unsigned long long *bb = nullptr;  // 2 x MAXD bbox words
  int cache_alloc_slots = 0;  // slots per cluster the cache tables were allocated for
  int64_t lay_n = 0;          // points in the current layout (all n for one instance)
  // pairs of at least this many point pairs go to the GPU-wide evaluation
  // (FP32 / FP64 values); HAC_BIG_PAIRS / HAC_BIG_PAIRS_F64 override them
  long long big_pairs = hacg::BIG_PAIRS, big_pairs64 = hacg::BIG_PAIRS_F64;
  long long warp_budget = hacg::WARP_BUDGET;  // HAC_WARP_BUDGET overrides it
  int brute_env = -1;   // HAC_BRUTE: -1 unset, 0 never, 1 whenever allowed
  // average linkage switches to the dense matrix once at most this many
  // clusters are active (HAC_DENSE_K overrides it; 0 = never)
  int64_t dense_k = -1;  // -1: the default for the instance
  int64_t dense_def = 0;  // that default for the current run (dense_default)
  int64_t dense_cap = 0; // matrix dimension the buffers were allocated for
  double *dense_buf = nullptr;  // the matrix buffers, dense_stride doubles each
  size_t dense_stride = 0;
  int dense_first = 0;   // the current run starts on the matrix
  int64_t dense_k0 = 0;  // active clusters when the run switched to the matrix
  // the point layout is older than the clusters: on the matrix points only
  // move when a re-score needs them (relayout_if_stale)
  int lay_stale = 0;
  int64_t launches = 0;  // kernels launched in the current run
  int ocur = 0, pcur = 0;
  bool done = false;
  int64_t n_merges = 0;
  hac_stats_t st{};
  // hac_run_static: memory for the packed triangle of up to tri_cap clusters
  // (filled once, from tri_k0 clusters)
  void *tri = nullptr;
  int tri_cap = 0, tri_k0 = 0;
  hac_merge *dout = nullptr;        // canonical dendrogram (device)
  int32_t *dout_round = nullptr;
};

namespace hacg {

template <typename T>
int dalloc(hac_ctx *h, T **p, size_t count) {
  if (count == 0) count = 1;
  void *q = nullptr;
  if (cudaMalloc(&q, count * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    return HAC_ENOMEM;
  }
  try {
    h->allocs.push_back(q);
  } catch (...) {
    cudaFree(q);
    return HAC_ENOMEM;
  }
  h->bytes += (int64_t)(count * sizeof(T));
  *p = (T *)q;
  return HAC_OK;
}

// Several arrays in one allocation: add() them all, then commit().  A handle
// holds about 75; one cudaMalloc and cudaFree each made 0.45 ms of a 0.63 ms
// hac.cluster of 64 points.
struct SlabAlloc {
  static constexpr int kMax = 96;
  static constexpr size_t kAlign = 256;
  void **at[kMax];
  size_t off[kMax];
  int n = 0;
  size_t bytes = 0;
  template <typename T>
  void add(T **p, size_t count) {
    if (n == kMax) {  // counted again by commit
      ++n;
      return;
    }
    at[n] = (void **)p;
    off[n++] = bytes;
    bytes += (std::max<size_t>(count, 1) * sizeof(T) + kAlign - 1) / kAlign * kAlign;
  }
  int commit(hac_ctx *h) {
    if (n > kMax) return HAC_EINTERNAL;
    unsigned char *q = nullptr;
    const int rc = dalloc(h, &q, bytes);
    if (rc) return rc;
    for (int i = 0; i < n; ++i) *at[i] = q + off[i];
    return HAC_OK;
  }
};

// Runs f() and turns a C++ exception (a failed host allocation, a thread
// that could not start) into a status code, so that none crosses the C ABI.
template <typename F>
int abi_guard(F &&f) noexcept {
  try {
    return f();
  } catch (const std::bad_alloc &) {
    return HAC_ENOMEM;
  } catch (...) {
    return HAC_EINTERNAL;
  }
}

void free_all(hac_ctx *h);
int pad_dim(int d);
int alloc_state(hac_ctx *h);

#define CK(x)                                \
  do {                                       \
    cudaError_t e_ = (x);                    \
    if (e_ != cudaSuccess) return HAC_EDEVICE; \
  } while (0)

// SM count of the current device (looked up once per device)
int device_sms();

// grid of a grid-stride kernel: one thread per work item, at most 64 blocks
// per SM
inline int grid_for(int64_t work, int tpb) {
  int64_t g = (work + tpb - 1) / tpb;
  if (g < 1) g = 1;
  const int64_t cap = (int64_t)device_sms() * 64;
  if (g > cap) g = cap;
  return (int)g;
}

// tree over the first K clusters of `order`; stable LSD radix sort of the
// first m keys/values in h->keys[0]/vals[0] (returns the buffer holding the
// result); bits needed for values up to maxval
int build_tree(hac_ctx *h, const int32_t *order, int K, cudaStream_t st);
int radix_sort(hac_ctx *h, int m, int bits, cudaStream_t st);
int bits_for(int64_t maxval);

// Per-round timing / counters of round_step (events may be null: no timing)
struct RoundCtl {
  cudaEvent_t e1 = nullptr, e2 = nullptr, eq0 = nullptr, eq1 = nullptr, eb0 = nullptr,
              eb1 = nullptr;
  double ms_query = 0, ms_big = 0;
  int64_t qlaunch = 0, big_launch = 0, searches = 0;
  int64_t naive = 0;  // terminals x (active clusters - 1), summed over rounds
  int big_iters = 0, big_reqs = 0;
  double ms_dense = 0;         // device time of the dense sweep
  int64_t dense_launches = 0;  // launches of the dense phase's kernels
  int64_t dense_rounds = 0;    // rounds run on the dense matrix
  int64_t dense_rechecks = 0;  // matrix entries re-scored in FP64
};

// Rounds of a closed-form linkage run in one launch (hac_finish.cu): from the
// active and terminal lists, or (raw set) from the input points
struct FinArgs {
  State s;
  int K, nterm, round;   // active clusters, terminals, first round
  int rounds_max;        // rounds to run at most (0 = to the end)
  int Kc;                // staged capacity (set by the launch)
  float scale;           // largest |coordinate| after recentring (not direct)
  const int32_t *order;  // active cids
  int32_t *order_out;    // where they go if the round limit stops the run
  const void *raw;       // direct: the input points
  int in_f32;            // their type
  hac_merge *out;        // direct: the dendrogram in canonical order, and
  int32_t *out_round;    //   each merge's round
  int n_rec;             // direct: records to write
};
int launch_finish(FinArgs &a, cudaStream_t st);
// the canonical order of at most FIN_MAX_K merge records in one block
int launch_rec_sort(const State &s, int m, hac_merge *out, int32_t *out_round, cudaStream_t st);

int round_step(hac_ctx *h, cudaStream_t st, int round, int K, int nterm, RoundCtl &ctl,
               int *npairs_out);

// big-pair evaluation of requests [r0, r0 + m) (hac_big*.cu): drop duplicate
// requests and build the tile schedule; run the evaluation kernels; fold the
// tiles and fill the cache tables and this round's result table
int big_prepare(const State &s, int r0, int m, cudaStream_t st);
int launch_big(const State &s, int r0, cudaStream_t st);
int big_finish(const State &s, int r0, int m, cudaStream_t st);
int launch_big_complete(const State &s, int r0, cudaStream_t st);
int launch_big_average(const State &s, int r0, cudaStream_t st);

// dense phase (hac_dense.cu): room for the matrix of K clusters (allocated if
// need be); whether this round should run on the matrix (entering it if
// needed); the nearest-neighbour search of the round's terminals on the matrix
// (with the FP64 re-score of near ties in the FP32 mode); the matrix after the
// round's merges (after the compaction, Kold clusters before); every remaining
// round in one launch, at most `limit` of them (0 = all)
int64_t dense_default(int64_t n, int d, int linkage, int prec);
int dense_reserve(hac_ctx *h, int K);
int dense_maybe_enter(hac_ctx *h, cudaStream_t st, int K, RoundCtl &ctl);
int dense_search(hac_ctx *h, cudaStream_t st, int K, int nterm, RoundCtl &ctl);
int dense_update(hac_ctx *h, cudaStream_t st, int round, int Kold, int K);
int dense_finish(hac_ctx *h, cudaStream_t st, int K, int nterm, int round, int64_t limit,
                 Counters *c);

// FP64 average / complete: the remaining rounds on the packed triangle, at most
// `limit` of them (0 = all); its bytes per pair
int tri_finish(hac_ctx *h, cudaStream_t st, int K, int nterm, int round, int64_t limit,
               Counters *c);
size_t tri_bytes(int linkage);

// points moved so that every cluster is one segment again, if they are not
int relayout_if_stale(hac_ctx *h, cudaStream_t st);

// one thread-block cluster of nct blocks (1 .. 16, a power of two; fewer if the
// device cannot place them) running kern(*args) on st
int launch_cluster(const void *kern, int nct, int threads, size_t smem, void *args,
                   cudaStream_t st);

}  // namespace hacg
