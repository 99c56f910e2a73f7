// PML and TVaR (Section IV-A names both as metrics derived from the YLT) as empirical order
// statistics: PML(RP) is the ceil(N/RP)-th largest year loss, TVaR(p) the mean of the
// ceil(N(1-p)) largest.  Exact selection on order-preserving 64-bit keys of the FP64 year losses,
// by sampled splitters:
//   1. every block sorts the same sampled keys of its row (one random position in each of 256 or
//      1,024 equal parts) and keeps as splitters those near the targets' expected places; then it
//      classes its slice of the row: above, equal to or between splitters (ties have classes of
//      their own).  Also the row sum.
//   2. from the class totals, each target's class; the keys of classes that are open intervals (2 N
//      per sampled key, on average) go to a list
//   3. one block per target finds its key in its list
//   4. TVaR targets: the sums of the values above the selected keys
// Few rows take one cooperative launch over every SM (k_sel_grid, bounded grid barriers between the
// steps); many rows a thread-block cluster each (k_sel_cluster, hardware barriers, and blocks that
// need half an SM, so that they run beside other streams' kernels); rows of at most 4,096 values
// one block each that sorts them whole (k_sel_small).
// Results are bit-exact copies of YLT entries (PML) and deterministic FP64 sums (TVaR, mean):
// fixed per-thread order, fixed warp and block trees, block partials combined in a fixed order.
//
// What it replaces: a cooperative radix select of 8-bit digits (4 to 8 passes over the row with a grid
// barrier each).  Kernel time of one call, 3 targets / 6 targets and the mean, us:
//   rows x values   1 x 1e3    1 x 3e4    1 x 1.5e5  1 x 1e6    1 x 5e6    8 x 1e5    16 x 2e5   64 x 2e5
//   radix select    23 / 30    31 / 39    36 / 48    60 / 82    161 / 225  44 / 68    89 / 145   394 / 557
//   this            15 / 16    31 / 38    31 / 40    43 / 62    99 / 128   35 / 43    50 / 72    93 / 124
// Few rows are bound by the steps' latencies (sorting the sample 4-7 us, a barrier 1.5 us, a pick 3 us,
// each pass over the row one L2 round trip), many rows by reading them three times.

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include <cooperative_groups.h>

#include "ara_device.cuh"
#include "ara_select_plan.h"

namespace ara {

constexpr int SEL_MAX_T = 16;
constexpr int SEL_WARPS = SEL_THREADS / 32;
constexpr int SEL_PICK = 4096;                   // list keys the pick keeps in shared memory
constexpr unsigned SFULL = 0xffffffffu;

struct SelTargets {
  int32_t n_t;                 // targets per layer
  int32_t n_rp;                // targets [0, n_rp) are PML ranks, the rest TVaR counts
  int64_t rank[SEL_MAX_T];     // 1-based rank from the top
};

__device__ __forceinline__ bool in_interval(uint64_t k, uint64_t lo, uint64_t hi) {
  return (k > lo || (lo == 0ull && k == 0ull)) && (k < hi || (hi == ~0ull && k == ~0ull));
}

// Scratch (one allocation; the part from err up to state is zero-filled before the launch).  Layers count
// from the first one of a launch group; G of them share the working parts at a time.
struct SelScratch {
  uint32_t* err;               // [1], behind the results
  uint32_t* count;             // [G][SEL_CLASSES] class totals
  uint32_t* n_list;            // [G][n_t] keys in each list
  uint32_t* bar;               // [G] grid-barrier counters
  uint32_t* count2;            // second round: [G][n_t][SEL_CLASSES], else null
  uint32_t* n_list2;           // second round: [G][n_t]
  SelState* state;             // [n_layers][n_t]
  uint64_t* list;              // [G][n_t][cap]
  double* psum;                // [G][n_t][blocks] block partials of the tail sums
  double* pmean;               // [G][blocks] block partials of the row sum
  // results, contiguous: out, mean, err
  double* out;                 // [n_layers][n_t] PML / TVaR
  double* mean;                // [n_layers]
  unsigned long long* gt;      // [n_layers][n_t] #{y > key}
  unsigned long long* eq;      // [n_layers][n_t] #{y == key}
  int64_t cap;
  int32_t sample;              // sampled keys per row
  uint32_t* ext_err;           // optional (nullptr): also gets DERR_TIMEOUT
  // optional caller outputs, written directly (nullptr: results stay in out / mean only)
  double* user_pml;            // [n_layers][n_rp]
  double* user_tvar;           // [n_layers][n_t - n_rp]
  double* user_mean;           // [n_layers]
};

static SelScratch carve(void* base, const SelPlan& y) {
  char* p = (char*)base;
  SelScratch s{};
  s.out = (double*)(p + y.off[0]);
  s.mean = s.out + (size_t)y.n_layers * y.n_t;
  s.err = (uint32_t*)(p + y.off[1]);
  s.count = (uint32_t*)(p + y.off[2]);
  s.n_list = (uint32_t*)(p + y.off[3]);
  s.bar = (uint32_t*)(p + y.off[4]);
  s.count2 = y.rounds > 1 ? (uint32_t*)(p + y.off[5]) : nullptr;
  s.n_list2 = (uint32_t*)(p + y.off[6]);
  s.state = (SelState*)(p + y.off[7]);
  s.list = (uint64_t*)(p + y.off[8]);
  s.psum = (double*)(p + y.off[9]);
  s.pmean = (double*)(p + y.off[10]);
  s.gt = (unsigned long long*)(p + y.off[11]);
  s.eq = (unsigned long long*)(p + y.off[12]);
  s.cap = y.lists.cap;
  s.sample = y.lists.sample;
  return s;
}

// Bitonic sort of m shared-memory keys (a power of two: 512 E, or for E = 2 any from 64), descending,
// by the whole block, E per thread in registers: thread l of warp w holds the keys 32 E w + 32 u + l,
// so steps of stride below 32 are shuffles, those below 32 E stay within the thread and only the wider
// ones go through shared memory.  (256 keys take 3.9 us, 1,024 6.7, one block alone on its SM.
// The loops are not unrolled: the code runs once per launch, and fetching it costs more than running it.)
template <int E>
__device__ __forceinline__ void sort_keys(uint64_t* a, int m) {
  const int lane = threadIdx.x & 31, i0 = 32 * E * (int)(threadIdx.x >> 5) + lane;
  const bool has = i0 < m;   // m is a multiple of 32 E: whole warps
  uint64_t x[E];
#pragma unroll
  for (int u = 0; u < E; ++u) x[u] = has ? a[i0 + 32 * u] : 0ull;
  auto take = [](uint64_t mine, uint64_t other, bool larger) { return (mine > other) == larger ? mine : other; };
  // key i keeps the larger of the pair (i, i ^ j) when i is its lower place in a descending run
  auto larger = [](int i, int j, int k) { return ((i & j) == 0) == ((i & k) == 0); };
#pragma unroll 1
  for (int k = 2; k <= m; k <<= 1) {
#pragma unroll 1
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (!has && j < 32 * E) continue;
      if (j >= 32 * E) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < E; ++u)
          if (has) a[i0 + 32 * u] = x[u];
        __syncthreads();
#pragma unroll
        for (int u = 0; u < E; ++u)
          if (has) x[u] = take(x[u], a[(i0 + 32 * u) ^ j], larger(i0 + 32 * u, j, k));
      } else if (j >= 32) {
#pragma unroll
        for (int d = 1; d < E; d <<= 1)
          if (j == 32 * d) {
#pragma unroll
            for (int u = 0; u < E; ++u)
              if (!(u & d)) {
                const uint64_t p = x[u], q = x[u | d];
                const bool swap = (p < q) == (((i0 + 32 * u) & k) == 0);
                x[u] = swap ? q : p;
                x[u | d] = swap ? p : q;
              }
          }
      } else {
#pragma unroll
        for (int u = 0; u < E; ++u)
          x[u] = take(x[u], __shfl_xor_sync(SFULL, x[u], j), larger(i0 + 32 * u, j, k));
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < E; ++u)
    if (has) a[i0 + 32 * u] = x[u];
  __syncthreads();
}

// Sum over the block by fixed trees; the result is valid in thread 0.  (Carrying the rounding errors
// along, in the trees alone, made a call of one short row 60 % slower: an FP64 operation has a long
// latency here.)
__device__ __forceinline__ double warp_add(double a, int from) {
#pragma unroll
  for (int o = 16; o; o >>= 1)
    if (o <= from) a = __dadd_rn(a, __shfl_down_sync(SFULL, a, o));
  return a;
}
__device__ __forceinline__ double block_sum(double a, double* wsum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  a = warp_add(a, 16);
  if (lane == 0) wsum[warp] = a;
  __syncthreads();
  if (warp == 0) a = warp_add(lane < SEL_WARPS ? wsum[lane] : 0.0, SEL_WARPS / 2);
  __syncthreads();
  return a;
}

// TVaR of m values: the sum of the gt values above the key v, and (m - gt) times v.
__device__ __forceinline__ double tvar_of(double above, int64_t m, unsigned long long gt, double v) {
  return (above + (double)(m - (int64_t)gt) * v) / (double)m;
}

__device__ __forceinline__ void put_result(const SelScratch& sc, const SelTargets& tg, int layer, int t, double r) {
  const int nt = tg.n_t;
  sc.out[(int64_t)layer * nt + t] = r;
  if (t < tg.n_rp) {
    if (sc.user_pml) sc.user_pml[(int64_t)layer * tg.n_rp + t] = r;
  } else if (sc.user_tvar) {
    sc.user_tvar[(int64_t)layer * (nt - tg.n_rp) + (t - tg.n_rp)] = r;
  }
}

__device__ __forceinline__ void put_mean(const SelScratch& sc, int layer, double r) {
  sc.mean[layer] = r;
  if (sc.user_mean) sc.user_mean[layer] = r;
}

__device__ __forceinline__ void sel_timeout(const SelScratch& sc) {
  *(volatile uint32_t*)sc.err = 1u;   // device or mapped host memory
  if (sc.ext_err) atomicOr(sc.ext_err, DERR_TIMEOUT);
}

// Sum of the values of the first n keys, by a fixed tree per 256 keys; valid in lane 0 of the warp.
__device__ __forceinline__ double warp_sum_keys(const uint64_t* sk, int n) {
  const int lane = threadIdx.x & 31;
  double a = 0.0;
  for (int i0 = lane; i0 < n; i0 += 256) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = i0 + 32 * u < n ? value_of(sk[i0 + 32 * u]) : 0.0;
#pragma unroll
    for (int d = 4; d; d >>= 1)
#pragma unroll
      for (int u = 0; u < d; ++u) v[u] = __dadd_rn(v[u], v[u + d]);
    a = __dadd_rn(a, v[0]);
  }
  return warp_add(a, 16);
}

// Rows of at most SEL_SMALL values, one block each: the sorted row gives every result directly, a warp
// to a target (they are chains of dependent shared loads).  Latency bounds it: six rows of
// 1,600 to 3,300 values in four calls take 92 us, 133 with every step of the sort in shared memory and
// the targets one after another over the block.
template <int E>
__global__ void __launch_bounds__(SEL_THREADS)
k_sel_small(const double* __restrict__ ylt, int32_t n, int32_t n_pad, SelTargets tg, SelScratch sc, int want_mean) {
  extern __shared__ uint64_t sk[];
  __shared__ double wsum[SEL_WARPS];
  const int layer = blockIdx.x, nt = tg.n_t, lane = threadIdx.x & 31;
  const double* src = ylt + (int64_t)layer * n;
  for (int i = threadIdx.x; i < n_pad; i += SEL_THREADS) sk[i] = i < n ? key_of(__ldcg(src + i)) : 0ull;
  __syncthreads();
  // keys are never 0 for the row's values except the NaN of all ones, which sorts with the padding
  sort_keys<E>(sk, n_pad);
  if (want_mean) {
    double a = 0.0;
    for (int i = threadIdx.x; i < n; i += SEL_THREADS) a = __dadd_rn(a, value_of(sk[i]));
    const double s = block_sum(a, wsum);
    if (threadIdx.x == 0) put_mean(sc, layer, s / (double)n);
  }
  for (int t = threadIdx.x >> 5; t < nt; t += SEL_WARPS) {
    const uint64_t key = sk[tg.rank[t] - 1];
    int lo = 0, hi = n;
    if (lane < 2)            // keys above (lane 0) and at or above (lane 1) the selected key
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (lane == 0 ? sk[mid] > key : sk[mid] >= key) lo = mid + 1;
        else hi = mid;
      }
    const int gt = __shfl_sync(SFULL, lo, 0), ge = __shfl_sync(SFULL, lo, 1);
    double r = value_of(key);
    if (t >= tg.n_rp) r = tvar_of(warp_sum_keys(sk, gt), tg.rank[t], (unsigned long long)gt, r);
    if (lane == 0) {
      put_result(sc, tg, layer, t, r);
      sc.gt[(int64_t)layer * nt + t] = (unsigned long long)gt;
      sc.eq[(int64_t)layer * nt + t] = (unsigned long long)(ge - gt);
      sc.state[(int64_t)layer * nt + t].key = key;
    }
  }
}

// ------------------------------------------------------------------------------------------
// The steps, for one block's slice of one row
// ------------------------------------------------------------------------------------------
constexpr int SEL_U = 4;                      // values per thread and step; the next ones are in flight
constexpr int SEL_QUEUE = 32 + 32 * SEL_U;    // keys a warp's queue can hold
struct SelShared {                            // shared memory of a block (dynamic: SEL_SMEM bytes)
  uint64_t key[SEL_SAMPLE];                   // the sorted sample, then the splitters
  uint64_t queue[SEL_WARPS][SEL_QUEUE];       // per warp: keys waiting for a full warp
  union {
    uint64_t keep[SEL_PICK];                  // the pick's list
    double psum[SEL_MAX_T][SEL_SLICES];       // afterwards, a cluster's block: its partial tail sums, by part
  };
  uint32_t hist[SEL_CLASSES];                 // class counts of the slice (the pick: digit counts)
  uint32_t cnt[SEL_CLASSES];                  // inclusive prefix of the row's class totals
  uint64_t ext[2 * SEL_WARPS];
  double wsum[SEL_WARPS];
  uint32_t wcnt[SEL_WARPS];
  SelState st[SEL_MAX_T];
  int32_t cls[SEL_MAX_T];
  uint64_t lo[SEL_MAX_T], width[SEL_MAX_T];   // the intervals to collect: keys lo .. lo + width
  int32_t own[SEL_MAX_T], n_own;
  uint32_t got[SEL_MAX_T], base[SEL_MAX_T];
  uint64_t found, prefix;
  int64_t k, gt, eq;
  // a cluster's row: its own partial row sums, by part, and (rank 0) the row's lists and picked targets
  double pmean[SEL_SLICES];
  uint32_t reported, n_list[SEL_MAX_T];
  uint64_t pick_key[SEL_MAX_T];
  int64_t pick_gt[SEL_MAX_T];
};
constexpr int SEL_SMEM = (int)sizeof(SelShared);

// Calls f(key, valid) for every key >= floor_key of the values [i0, i1) of the row: such keys wait in
// the warp's queue until 32 are there, so f runs on full warps however few they are (all lanes
// call it; the last call may have invalid lanes).  all(y, u) sees every value in order (0 past the
// slice's end; u: 0 .. 3 in turn).  The order of the calls depends on the row alone.  f appears once:
// the code runs once or twice per launch, and fetching it costs more than running it.  Returns
// the number of keys >= floor_key (per warp).
template <typename F, typename G>
__device__ __forceinline__ uint32_t for_keys_from(const double* __restrict__ row, int64_t i0, int64_t i1,
                                                  uint64_t floor_key, uint64_t* q, F&& f, G&& all) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int qn = 0;
  uint32_t total = 0;
  double next[SEL_U];
  const double* at = row + i0 + threadIdx.x;
  int64_t left = i1 - i0 - (int64_t)threadIdx.x;   // values from this thread's place to the end
#pragma unroll
  for (int u = 0; u < SEL_U; ++u) next[u] = left > u * SEL_THREADS ? __ldcg(at + u * SEL_THREADS) : 0.0;
  bool more = true;
  while (more) {
    double y[SEL_U];
    const int64_t here = left;
    at += SEL_U * SEL_THREADS;
    left -= SEL_U * SEL_THREADS;
    more = left + lane > 0;                        // uniform over the warp
#pragma unroll
    for (int u = 0; u < SEL_U; ++u) {
      y[u] = next[u];
      next[u] = left > u * SEL_THREADS ? __ldcg(at + u * SEL_THREADS) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < SEL_U; ++u) {
      if (here + lane <= u * SEL_THREADS) break;   // uniform: the warp is past the end
      all(y[u], u);
      const uint64_t k = key_of(y[u]);
      const bool c = here > u * SEL_THREADS && k >= floor_key;
      const unsigned m = __ballot_sync(SFULL, c);
      if (c) q[qn + __popc(m & lt)] = k;
      qn += __popc(m);
    }
    __syncwarp();
#pragma unroll 1
    while (qn >= 32 || (!more && qn > 0)) {
      const int n = min(qn, 32);
      qn -= n;
      total += (uint32_t)n;
      f(lane < n ? q[qn + lane] : 0ull, lane < n);
    }
    __syncwarp();
  }
  return total;
}

// The row's splitters into S.key (descending); returns their number.  With a list (of cap keys):
// SEL_SAMPLE keys of it, all of them.
__device__ __forceinline__ int row_splitters(SelShared& S, const double* __restrict__ row, int64_t n, int sample,
                                             const SelTargets& tg, const uint64_t* list = nullptr, int64_t cap = 0) {
  const int nt = tg.n_t, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (list) sample = SEL_SAMPLE;
  const int lg = 31 - __clz(sample);   // a power of two
  for (int j = threadIdx.x; j < sample; j += SEL_THREADS) {
    const int64_t a = ((int64_t)j * n) >> lg, b = ((int64_t)(j + 1) * n) >> lg;
    uint64_t z = (uint64_t)(j + 1) * 0x9E3779B97F4A7C15ull;   // SplitMix64 of the part's number
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    S.key[j] = list ? __ldcg(list + (((int64_t)j * cap) >> lg))
                    : key_of(__ldcg(row + a + (int64_t)__umul64hi(z, (uint64_t)(b - a))));
  }
  __syncthreads();
  sort_keys<2>(S.key, sample);
  if (list) return sample;
  // Splitters: sample places within 6 standard deviations (and 4 places) of a target's expected
  // place.  Kept places move to the front in order.
  bool keep[SEL_SAMPLE / SEL_THREADS];
  uint64_t mine[SEL_SAMPLE / SEL_THREADS];
#pragma unroll
  for (int u = 0; u < SEL_SAMPLE / SEL_THREADS; ++u) {
    const int i = u * SEL_THREADS + (int)threadIdx.x;
    mine[u] = S.key[i];
    keep[u] = false;
    for (int t = 0; t < nt && i < sample; ++t) {
      const float r = (float)tg.rank[t] * ((float)sample / (float)n);
      const float w = 6.0f * sqrtf(fmaxf(r * (1.0f - r / (float)sample), 1.0f)) + 4.0f;
      keep[u] = keep[u] || fabsf((float)i - r) <= w;
    }
  }
  __syncthreads();
  int np = 0;
#pragma unroll
  for (int u = 0; u < SEL_SAMPLE / SEL_THREADS; ++u) {
    const unsigned m = __ballot_sync(SFULL, keep[u]);
    if (lane == 0) S.wcnt[warp] = (uint32_t)__popc(m);
    __syncthreads();
    int at = np, all = np;
    for (int w = 0; w < SEL_WARPS; ++w) {
      if (w < warp) at += (int)S.wcnt[w];
      all += (int)S.wcnt[w];
    }
    if (keep[u]) S.key[at + __popc(m & ((1u << lane) - 1u))] = mine[u];
    np = all;
    __syncthreads();
  }
  return np;
}

// Part v of V of a row of n values.
__device__ __forceinline__ int64_t slice_begin(int64_t n, unsigned v, unsigned V) { return (int64_t)v * n / V; }

// Class counts of the row's parts [v0, v1) of V into S.hist.  Class 2 i: between splitters i - 1 and i;
// class 2 i + 1: equal to splitter i (its first place).  Only keys within [lo, hi] count (the whole range,
// or an interval that is split again).  out(v, sum) is called by thread 0 for each part when want_mean.
// PARTS: there may be more than one part.
template <bool PARTS, typename O>
__device__ __forceinline__ void count_slices(SelShared& S, const double* __restrict__ row, int64_t n, unsigned v0,
                                             unsigned v1, unsigned V, int np, uint64_t lo, uint64_t hi, int want_mean,
                                             O&& out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i <= 2 * np; i += SEL_THREADS) S.hist[i] = 0u;
  __syncthreads();
  const int top = np > 0 ? 1 << (31 - __clz(np)) : 0;
  const bool part = lo != 0ull || hi != ~0ull;
  // keys below every splitter are counted, not searched
  const uint64_t floor_key = np == 0 ? ~0ull : part ? lo : S.key[np - 1];
  uint32_t near = 0;
  unsigned v = v0;
  do {
    double sum[2] = {0.0, 0.0};
    near += for_keys_from(row, slice_begin(n, v, V), slice_begin(n, v + 1, V), floor_key, S.queue[warp], [&](uint64_t k, bool valid) {
      if (part) valid = valid && in_interval(k, lo, hi);
      int c = 0;               // splitters above k
      for (int step = top; step; step >>= 1)
        if (c + step <= np && S.key[c + step - 1] > k) c += step;
      const uint32_t cls = valid ? 2u * (uint32_t)c + (np > 0 && S.key[min(c, np - 1)] == k ? 1u : 0u) : 0xffffffffu;
      const unsigned peers = __match_any_sync(SFULL, cls);
      if (valid && lane == __ffs(peers) - 1) atomicAdd(&S.hist[cls], (uint32_t)__popc(peers));
    }, [&](double y, int u) {
      if (want_mean) sum[u & 1] = __dadd_rn(sum[u & 1], y);
    });
    if (want_mean) {
      const double s = block_sum(__dadd_rn(sum[0], sum[1]), S.wsum);
      if (threadIdx.x == 0) out(v, s);
    }
  } while (PARTS && ++v < v1);
  if (lane == 0) S.wcnt[warp] = near;
  __syncthreads();
  if (warp == 0 && np > 0 && !part) {
    const uint32_t counted = __reduce_add_sync(SFULL, lane < SEL_WARPS ? S.wcnt[lane] : 0u);
    if (lane == 0) S.hist[2 * np] += (uint32_t)(slice_begin(n, v1, V) - slice_begin(n, v0, V)) - counted;
  }
  __syncthreads();
}

// The classes of the targets [first, last) from the row's class totals (S.cnt, i <= 2 np; a barrier
// after they were written), into S.st, and the intervals to collect (S.own, S.lo, S.width; one per distinct class).  old: the
// interval that was split (the whole range at first), with the keys before it.
__device__ __forceinline__ void target_classes(SelShared& S, const SelTargets& tg, int first, int last, int np,
                                               uint64_t old_lo, uint64_t old_hi, int64_t old_before) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (2 * np + SEL_THREADS) / SEL_THREADS;   // classes per thread
  uint32_t s = 0;
  for (int u = 0; u < per; ++u) {
    const int i = (int)threadIdx.x * per + u;
    s += i <= 2 * np ? S.cnt[i] : 0u;
  }
  uint32_t incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(SFULL, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31) S.wcnt[warp] = incl;
  __syncthreads();
  uint32_t run = incl - s;
  for (int w = 0; w < warp; ++w) run += S.wcnt[w];
  for (int u = 0; u < per; ++u) {
    const int i = (int)threadIdx.x * per + u;
    if (i <= 2 * np) {
      run += S.cnt[i];
      S.cnt[i] = run;
    }
  }
  __syncthreads();
  const int q = first + (int)threadIdx.x;
  if (q < last) {            // the first class whose prefix reaches the rank
    const int64_t k = tg.rank[q] - old_before;
    int a = 0, b = 2 * np;
    while (a < b) {
      const int mid = (a + b) >> 1;
      if ((int64_t)S.cnt[mid] >= k) b = mid;
      else a = mid + 1;
    }
    const int64_t before = a ? (int64_t)S.cnt[a - 1] : 0;
    const int i = a >> 1;    // class 2 i: above splitter i (if any) and below splitter i - 1 (if any)
    S.st[q] = SelState{a & 1 ? S.key[i] : 0ull, i < np ? S.key[i] : old_lo, i > 0 ? S.key[i - 1] : old_hi,
                       a & 1, q, old_before + before, (int64_t)S.cnt[a] - before};
    S.cls[q] = a;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int m = 0;
    for (int t = first; t < last; ++t) {
      int f = first;
      while (S.cls[f] != S.cls[t]) ++f;
      S.st[t].list = f;
      if (f == t && !S.st[t].tie) {
        const uint64_t l = S.st[t].lo, h = S.st[t].hi;
        S.own[m] = t;
        S.lo[m] = l == 0ull ? 0ull : l + 1;
        S.width[m] = (h == ~0ull ? h : h - 1) - S.lo[m];
        ++m;
      }
    }
    S.n_own = m;
  }
  __syncthreads();
}

// The slice's keys of the intervals, appended to the targets' lists (of at most cap keys); counter(t)
// is the address of target t's list length.
template <typename C>
__device__ __forceinline__ void collect_slice(SelShared& S, const double* __restrict__ row, int64_t i0, int64_t i1,
                                              uint64_t* list, int64_t cap, C&& counter) {
  const int m = S.n_own, warp = threadIdx.x >> 5;
  if (m == 0) return;
  uint64_t floor_key = ~0ull;
  for (int q = 0; q < m; ++q) floor_key = min(floor_key, S.lo[q]);
  // First into the block's own part of S.keep, then to the list with one reservation per interval; what
  // the part does not hold goes there directly.
  const int part = SEL_PICK / m;
  if (threadIdx.x < SEL_MAX_T) S.got[threadIdx.x] = 0u;
  __syncthreads();
  for_keys_from(row, i0, i1, floor_key, S.queue[warp], [&](uint64_t k, bool valid) {
    int mine = -1;           // the intervals are disjoint
    for (int q = 0; q < m; ++q)
      if (valid && k - S.lo[q] <= S.width[q]) mine = q;
    if (mine < 0) return;
    const uint32_t at = atomicAdd(&S.got[mine], 1u);
    if (at < (uint32_t)part) {
      S.keep[mine * part + (int)at] = k;
    } else {
      const int t = S.own[mine];
      const uint32_t p = atomicAdd(counter(t), 1u);
      if ((int64_t)p < cap) list[(int64_t)t * cap + p] = k;
    }
  }, [](double, int) {});
  __syncthreads();
  if (threadIdx.x < m) {
    const uint32_t c = min(S.got[threadIdx.x], (uint32_t)part);
    S.got[threadIdx.x] = c;
    S.base[threadIdx.x] = c ? atomicAdd(counter(S.own[threadIdx.x]), c) : 0u;
  }
  __syncthreads();
  for (int q = 0; q < m; ++q)
    for (uint32_t i = threadIdx.x; i < S.got[q]; i += SEL_THREADS) {
      const int64_t at = (int64_t)S.base[q] + i;
      if (at < cap) list[(int64_t)S.own[q] * cap + at] = S.keep[q * part + (int)i];
    }
  __syncthreads();
}

// The key of rank `rank` of a target with state st, by the whole block; *gt and *eq: keys above and
// equal to it.  list: the list of its interval; one that did not fit is replaced by the row's keys.
__device__ __forceinline__ uint64_t pick_key(SelShared& S, const double* __restrict__ row, int64_t n, const SelState& st,
                                             int64_t rank, const uint64_t* list, int64_t cap, int64_t* gt, int64_t* eq) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (st.tie) {
    *gt = st.before;
    *eq = st.in_class;
    return st.key;
  }
  const bool listed = st.in_class <= cap;
  const int64_t N = listed ? st.in_class : n;
  const bool near = listed && N <= SEL_PICK;
  auto get = [&](int64_t i, bool& in) -> uint64_t {
    in = true;
    if (near) return S.keep[i];
    if (listed) return __ldcg(list + i);
    const uint64_t k = key_of(__ldcg(row + i));
    in = in_interval(k, st.lo, st.hi);
    return k;
  };
  if (listed && N <= 192) {   // short lists (the counting grows with their square): every thread counts the keys above its own
    const int c = (int)N;
    const uint64_t x = (int)threadIdx.x < c ? __ldcg(list + threadIdx.x) : 0ull;
    if ((int)threadIdx.x < c) S.keep[threadIdx.x] = x;
    __syncthreads();
    if ((int)threadIdx.x < c) {
      int above = 0, same = 0;
#pragma unroll 2
      for (int i = 0; i < c; ++i) {
        const uint64_t o = S.keep[i];
        above += o > x ? 1 : 0;
        same += o == x ? 1 : 0;
      }
      const int64_t k = rank - st.before;
      if (above < k && k <= above + same) {   // the threads of equal keys write the same values
        S.found = x;
        S.gt = above;
        S.eq = same;
      }
    }
    __syncthreads();
    const uint64_t key = S.found;
    *gt = st.before + S.gt;
    *eq = S.eq;
    __syncthreads();
    return key;
  }
  // the highest bit in which the keys differ
  uint64_t mn = ~0ull, mx = 0ull;
  for (int64_t i = threadIdx.x; i < N; i += SEL_THREADS) {
    bool in = true;
    uint64_t k;
    if (near) S.keep[i] = k = __ldcg(list + i);
    else k = get(i, in);
    if (in) { mn = min(mn, k); mx = max(mx, k); }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    mn = min(mn, (uint64_t)__shfl_xor_sync(SFULL, mn, o));
    mx = max(mx, (uint64_t)__shfl_xor_sync(SFULL, mx, o));
  }
  if (lane == 0) { S.ext[warp] = mn; S.ext[SEL_WARPS + warp] = mx; }
  __syncthreads();
  for (int w = 0; w < SEL_WARPS; ++w) {
    mn = min(mn, S.ext[w]);
    mx = max(mx, S.ext[SEL_WARPS + w]);
  }
  // radix select on 8-bit digits, from the first digit that differs until one key is left
  const uint64_t diff = mn ^ mx;
  int shift = diff ? (63 - __clzll((long long)diff)) / 8 * 8 : 0;
  uint64_t prefix = mx >> shift >> 8;                // the bits above the digit
  int64_t k = rank - st.before, above = 0, count = 0;
  while (true) {
    for (int i = threadIdx.x; i < 256; i += SEL_THREADS) S.hist[i] = 0u;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < N; i += SEL_THREADS) {
      bool in;
      const uint64_t x = get(i, in);
      if (in && (x >> shift >> 8) == prefix) atomicAdd(&S.hist[(x >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (warp == 0) {         // lane l owns bins [256 - 8 (l + 1), 256 - 8 l), from the top down
      uint32_t h[8], mine = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        h[u] = S.hist[255 - (8 * lane + u)];
        mine += h[u];
      }
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(SFULL, incl, o);
        if (lane >= o) incl += x;
      }
      const int64_t excl = (int64_t)(incl - mine);
      if (excl < k && k <= (int64_t)incl) {
        int64_t b4 = excl;
        int u = 0;
        for (; u < 7; ++u) {
          if (b4 + h[u] >= k) break;
          b4 += h[u];
        }
        S.prefix = (prefix << 8) | (uint64_t)(255 - (8 * lane + u));
        S.k = k - b4;
        S.gt = above + b4;
        S.eq = h[u];
      }
    }
    __syncthreads();
    prefix = S.prefix;       // down to and including this digit
    k = S.k;
    above = S.gt;
    count = S.eq;
    __syncthreads();
    if (count == 1 || shift == 0) break;
    shift -= 8;
  }
  uint64_t key = prefix;
  if (shift > 0) {           // one key has this prefix
    for (int64_t i = threadIdx.x; i < N; i += SEL_THREADS) {
      bool in;
      const uint64_t x = get(i, in);
      if (in && (x >> shift) == prefix) S.found = x;
    }
    __syncthreads();
    key = S.found;
    __syncthreads();
  }
  *gt = st.before + above;
  *eq = count;
  return key;
}

// The slice's sums of the values above thr[q], q < m <= 4; out(q, sum) is called by thread 0.
template <typename O>
__device__ __forceinline__ void tail_slice(SelShared& S, const double* __restrict__ row, int64_t i0, int64_t i1, int m,
                                           const uint64_t (&thr)[4], O&& out) {
  uint64_t least = ~0ull;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int q = 0; q < 4; ++q) least = q < m ? min(least, thr[q]) : least;
  for_keys_from(row, i0, i1, least, S.queue[threadIdx.x >> 5], [&](uint64_t k, bool valid) {
    const double y = value_of(k);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < m && valid && k > thr[q]) a[q] = __dadd_rn(a[q], y);
  }, [](double, int) {});
#pragma unroll 1
  for (int q = 0; q < m; ++q) {
    const double s = block_sum(q == 0 ? a[0] : q == 1 ? a[1] : q == 2 ? a[2] : a[3], S.wsum);
    if (threadIdx.x == 0) out(q, s);
  }
}

// ------------------------------------------------------------------------------------------
// One kernel per row in a thread-block cluster: the steps with cluster barriers between them.
// ------------------------------------------------------------------------------------------
// PARTS: the row's sums are taken in V parts, several to a block, as the cooperative form takes them, so
// that both give the same bits (a burst of 12 served requests takes 0.4 to 0.9 % longer for it); otherwise V
// is the number of blocks.
template <bool PARTS>
__global__ void __launch_bounds__(SEL_THREADS, 2)
k_sel_cluster(const double* __restrict__ ylt, int64_t n, int32_t l0, unsigned n_parts, SelTargets tg, SelScratch sc,
              int want_mean, int skip_report) {
  extern __shared__ __align__(16) unsigned char sel_smem[];
  SelShared& S = *reinterpret_cast<SelShared*>(sel_smem);
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned B = gridDim.x, rank = blockIdx.x;     // a cluster spans the grid's x
  const int layer = l0 + (int)blockIdx.y, nt = tg.n_t;
  const double* row = ylt + (int64_t)layer * n;
  const unsigned V = PARTS ? n_parts : B;
  const unsigned v0 = PARTS ? rank * V / B : rank, v1 = PARTS ? (rank + 1) * V / B : rank + 1;   // this block's parts
  const int64_t i0 = slice_begin(n, v0, V), i1 = slice_begin(n, v1, V);
  if (threadIdx.x < SEL_MAX_T) S.n_list[threadIdx.x] = 0u;
  const int np = nt > 0 ? row_splitters(S, row, n, sc.sample, tg) : 0;
  count_slices<PARTS>(S, row, n, v0, v1, V, np, 0ull, ~0ull, want_mean, [&](unsigned v, double s) { S.pmean[v - v0] = s; });
  if (threadIdx.x == 0) S.reported = skip_report ? 0u : 1u;
  cluster.sync();
  // (remote words are read by different threads at once: one after the other costs 300 cycles each)
  const unsigned lane = threadIdx.x & 31;
  const bool ok = __all_sync(SFULL, lane >= B || cluster.map_shared_rank(&S, lane < B ? lane : 0u)->reported != 0u);
  if (ok && nt > 0) {
    for (int i = threadIdx.x; i <= 2 * np; i += SEL_THREADS) S.cnt[i] = 0u;
    __syncthreads();
    const unsigned shift = 31u - (unsigned)__clz((int)B);   // B is a power of two
    for (unsigned i = threadIdx.x; i < (unsigned)(2 * np + 1) << shift; i += SEL_THREADS) {
      const uint32_t v = cluster.map_shared_rank(&S, i & (B - 1u))->hist[i >> shift];
      if (v) atomicAdd(&S.cnt[i >> shift], v);
    }
    __syncthreads();
    target_classes(S, tg, 0, nt, np, 0ull, ~0ull, 0);
    SelShared* const head = cluster.map_shared_rank(&S, 0);
    collect_slice(S, row, i0, i1, sc.list + (int64_t)layer * nt * sc.cap, sc.cap,
                  [&](int t) -> uint32_t* { return &head->n_list[t]; });
  }
  cluster.sync();                                      // lists complete, class counts read
  if (ok) {
    SelShared* const head = cluster.map_shared_rank(&S, 0);
    for (int t = (int)rank; t < nt; t += (int)B) {
      const SelState st = S.st[t];
      int64_t gt, eq;
      const uint64_t key = pick_key(S, row, n, st, tg.rank[t], sc.list + ((int64_t)layer * nt + st.list) * sc.cap,
                                    sc.cap, &gt, &eq);
      if (threadIdx.x == 0) {
        const int64_t lt = (int64_t)layer * nt + t;
        head->pick_key[t] = key;
        head->pick_gt[t] = gt;
        sc.state[lt].key = key;
        sc.gt[lt] = (unsigned long long)gt;
        sc.eq[lt] = (unsigned long long)eq;
        if (t < tg.n_rp) put_result(sc, tg, layer, t, value_of(key));
      }
    }
  }
  cluster.sync();                                      // every target's key is in rank 0
  if (ok)
    for (int t0 = tg.n_rp; t0 < nt; t0 += 4) {
      uint64_t thr[4];
      const int m = min(4, nt - t0);
#pragma unroll
      for (int q = 0; q < 4; ++q) thr[q] = q < m ? cluster.map_shared_rank(&S, 0)->pick_key[t0 + q] : ~0ull;
      unsigned v = v0;
      do {
        tail_slice(S, row, PARTS ? slice_begin(n, v, V) : i0, PARTS ? slice_begin(n, v + 1, V) : i1, m, thr,
                   [&](int q, double s) { S.psum[t0 + q][v - v0] = s; });
      } while (PARTS && ++v < v1);
    }
  cluster.sync();                                      // partial sums complete
  if (rank == 0) {
    // warp w: result w of the mean (if wanted) and the TVaR targets, from the parts' sums by the tree of
    // block_sum over one part per thread
    if (!ok && threadIdx.x == 0) sel_timeout(sc);
    for (int w = (int)(threadIdx.x >> 5); ok && w < 1 + nt - tg.n_rp; w += SEL_WARPS) {
      if (w == 0 && !want_mean) continue;
      const int t = tg.n_rp + w - 1;
      double a;
      if constexpr (!PARTS) {     // one part to a block (with the loop below, 16 targets took 7 % longer)
        const SelShared* const o = cluster.map_shared_rank(&S, lane < B ? lane : 0u);
        a = warp_add(lane < B ? (w == 0 ? o->pmean[0] : o->psum[t][0]) : 0.0, 8);
      } else {
        double wsum = 0.0;                             // lane l: the sum of the parts 32 l .. 32 l + 31
        for (unsigned base = 0; base < V; base += 32) {
          const unsigned v = base + lane;
          double x = 0.0;
          if (v < V) {
            const unsigned owner = ((v + 1) * B - 1) / V;
            const SelShared* const o = cluster.map_shared_rank(&S, owner);
            const unsigned at = v - owner * V / B;
            x = w == 0 ? o->pmean[at] : o->psum[t][at];
          }
          const double sum = __shfl_sync(SFULL, warp_add(x, 16), 0);
          if (lane == base / 32) wsum = sum;
        }
        a = warp_add(lane < SEL_WARPS ? wsum : 0.0, SEL_WARPS / 2);
      }
      if (lane != 0) continue;
      if (w == 0) {
        put_mean(sc, layer, a / (double)n);
      } else {
        put_result(sc, tg, layer, t, tvar_of(a, tg.rank[t], (unsigned long long)S.pick_gt[t], value_of(S.pick_key[t])));
      }
    }
  }
  cluster.sync();                                      // no block leaves while rank 0 reads it
}

// ------------------------------------------------------------------------------------------
// Few rows: the steps in one cooperative launch over every SM, the blocks of a row meeting at grid
// barriers (bounded waits).
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t sel_globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Every block adds one to *bar, then waits until it reaches `target` (the number of blocks times the
// barrier's ordinal).  The wait is bounded by limit_ns; on timeout the block records it and the
// whole block returns false.
__device__ __forceinline__ bool grid_barrier(uint32_t* bar, uint32_t target, uint64_t limit_ns, const SelScratch& sc,
                                             int skip_arrival, int* ok_s) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (!skip_arrival) atomicAdd(bar, 1u);
    int ok = 1;
    if (ld_acquire_gpu(bar) < target) {
      const uint64_t t0 = sel_globaltimer();
      while (ld_acquire_gpu(bar) < target) {
        if (sel_globaltimer() - t0 > limit_ns) {
          ok = 0;
          sel_timeout(sc);
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
    *ok_s = ok;
  }
  __syncthreads();
  return *ok_s != 0;
}

__global__ void __launch_bounds__(SEL_THREADS, 2)
k_sel_grid(const double* __restrict__ ylt, int64_t n, int32_t l0, SelTargets tg, SelScratch sc, int want_mean,
           uint64_t limit_ns, int skip_arrival) {
  extern __shared__ __align__(16) unsigned char sel_smem[];
  SelShared& S = *reinterpret_cast<SelShared*>(sel_smem);
  __shared__ int ok_s;
  const unsigned B = gridDim.x;
  const int layer = l0 + (int)blockIdx.y, nt = tg.n_t;
  const int64_t lt0 = (int64_t)layer * nt;
  const double* row = ylt + (int64_t)layer * n;
  const int64_t i0 = slice_begin(n, blockIdx.x, B), i1 = slice_begin(n, blockIdx.x + 1, B);
  uint32_t met = 0;
  auto meet = [&]() { return grid_barrier(sc.bar + layer, ++met * B, limit_ns, sc, skip_arrival, &ok_s); };
  auto block_sums = [&](const double* p) {
    double a = 0.0;
    for (unsigned b = threadIdx.x; b < B; b += SEL_THREADS) a = __dadd_rn(a, __ldcg(p + b));
    return block_sum(a, S.wsum);
  };
  // Round t = nt: all targets.  Then, where lists may overflow (sc.count2), a round for each target
  // whose list did: its interval is split again by keys that made it into the list.  Every block
  // knows the same states.  A list is its first target's: the others sharing it go first.
#pragma unroll 1
  for (int t = nt; t >= 0; --t) {
    SelState old{0ull, 0ull, ~0ull, 0, 0, 0, 0};
    int np = 0;
    uint32_t *g = sc.count + (int64_t)layer * SEL_CLASSES, *n_list = sc.n_list + lt0;
    if (t < nt) {
      if (!sc.count2) break;
      old = S.st[t];
      if (old.tie || old.in_class <= sc.cap) continue;
      g = sc.count2 + (lt0 + t) * SEL_CLASSES;
      n_list = sc.n_list2 + lt0;
    }
    if (nt > 0) np = row_splitters(S, row, n, sc.sample, tg, t < nt ? sc.list + (lt0 + old.list) * sc.cap : nullptr, sc.cap);
    count_slices<false>(S, row, n, blockIdx.x, blockIdx.x + 1, B, np, old.lo, old.hi, t == nt ? want_mean : 0,
                 [&](unsigned b, double s) { sc.pmean[(int64_t)layer * B + b] = s; });
    for (int i = threadIdx.x; np > 0 && i <= 2 * np; i += SEL_THREADS)
      if (S.hist[i]) atomicAdd(g + i, S.hist[i]);
    if (!meet()) return;
    if (t == nt && want_mean && blockIdx.x == B - 1) {
      const double s = block_sums(sc.pmean + (int64_t)layer * B);
      if (threadIdx.x == 0) put_mean(sc, layer, s / (double)n);
    }
    if (nt == 0) return;
    for (int i = threadIdx.x; i <= 2 * np; i += SEL_THREADS) S.cnt[i] = __ldcg(g + i);
    __syncthreads();
    target_classes(S, tg, t < nt ? t : 0, t < nt ? t + 1 : nt, np, old.lo, old.hi, old.before);
    collect_slice(S, row, i0, i1, sc.list + lt0 * sc.cap, sc.cap, [&](int q) { return n_list + q; });
    if (!meet()) return;
  }
  for (int t = (int)blockIdx.x; t < nt; t += (int)B) {
    const SelState st = S.st[t];
    int64_t gt, eq;
    const uint64_t key = pick_key(S, row, n, st, tg.rank[t], sc.list + (lt0 + st.list) * sc.cap, sc.cap, &gt, &eq);
    if (threadIdx.x == 0) {
      sc.state[lt0 + t].key = key;
      sc.gt[lt0 + t] = (unsigned long long)gt;
      sc.eq[lt0 + t] = (unsigned long long)eq;
      if (t < tg.n_rp) put_result(sc, tg, layer, t, value_of(key));
    }
  }
  if (nt == tg.n_rp) return;
  if (!meet()) return;
  for (int t0 = tg.n_rp; t0 < nt; t0 += 4) {
    uint64_t thr[4];
    const int m = min(4, nt - t0);
#pragma unroll
    for (int q = 0; q < 4; ++q) thr[q] = q < m ? __ldcg(&sc.state[lt0 + t0 + q].key) : ~0ull;
    tail_slice(S, row, i0, i1, m, thr, [&](int q, double s) { sc.psum[(lt0 + t0 + q) * B + blockIdx.x] = s; });
  }
  if (!meet()) return;
  for (int t = tg.n_rp + (int)blockIdx.x; t < nt; t += (int)B) {
    const double s = block_sums(sc.psum + (lt0 + t) * B);
    if (threadIdx.x == 0)
      put_result(sc, tg, layer, t, tvar_of(s, tg.rank[t], __ldcg(sc.gt + lt0 + t), value_of(__ldcg(&sc.state[lt0 + t].key))));
  }
}

// ceil(x), taking x within 1e-9 (relative) of an integer as that integer.
static int64_t ceil_snap(double x) {
  const double r = std::nearbyint(x);
  if (std::fabs(x - r) <= 1e-9 * std::fmax(1.0, std::fabs(x))) return (int64_t)r;
  return (int64_t)std::ceil(x);
}

ara_status select_targets(int64_t n, int32_t n_rp, const double* rps, int32_t n_tvar,
                          const double* levels, SelTargets& tg) {
  if (n < 1 || n_rp < 0 || n_tvar < 0 || n_rp + n_tvar > SEL_MAX_T) return ARA_EINVAL;
  if ((n_rp > 0 && !rps) || (n_tvar > 0 && !levels)) return ARA_EINVAL;
  tg.n_t = n_rp + n_tvar;
  tg.n_rp = n_rp;
  for (int i = 0; i < n_rp; ++i) {
    if (!(rps[i] >= 1.0) || !std::isfinite(rps[i])) return ARA_EINVAL;
    const int64_t k = ceil_snap((double)n / rps[i]);
    if (k < 1 || k > n) return ARA_EINVAL;
    tg.rank[i] = k;
  }
  for (int i = 0; i < n_tvar; ++i) {
    if (!(levels[i] >= 0.0 && levels[i] < 1.0)) return ARA_EINVAL;
    const int64_t m = ceil_snap((double)n * (1.0 - levels[i]));
    if (m < 1 || m > n) return ARA_EINVAL;
    tg.rank[n_rp + i] = m;
  }
  return ARA_OK;
}

int64_t tail_count_snap(int64_t n, double p) {
  if (!(p >= 0.0 && p < 1.0) || n < 1) return -1;
  const int64_t m = ceil_snap((double)n * (1.0 - p));
  return (m >= 1 && m <= n) ? m : -1;
}

ara_status validate_metrics(int64_t n, int32_t n_rp, const double* rps, int32_t n_tvar,
                            const double* levels) {
  SelTargets tg;
  return select_targets(n, n_rp, rps, n_tvar, levels, tg);
}

// Shared-memory and cluster attributes of the kernels, set once per context.
static ara_status sel_prepare_kernels() {
  static std::mutex mu;
  static uint64_t done[64] = {0};
  int dev = 0;
  ARA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return ARA_ECUDA;
  const uint64_t ctx = context_id();
  std::lock_guard<std::mutex> lk(mu);
  if (ctx != 0 && done[dev] == ctx) return ARA_OK;
  for (const void* f : {(const void*)k_sel_cluster<false>, (const void*)k_sel_cluster<true>, (const void*)k_sel_grid})
    ARA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, SEL_SMEM));
  // k_sel_grid has at most one block per SM.  100 KB of shared memory (44 % of 228) keeps two from
  // sharing one while others stand empty, and a stream kernel queued behind it on another stream from
  // being given all 228 KB, which leaves its gathers little L1: the paper-scale step, selection on a
  // second stream, 1.167 -> 1.067 ms (selection 72 -> 61 us, stream 1.09 -> 1.00).
  ARA_TRY(cudaFuncSetAttribute((const void*)k_sel_grid, cudaFuncAttributePreferredSharedMemoryCarveout, 44));
  static_assert(SEL_SMEM <= 99 * 1024 && 2 * SEL_SMEM > 99 * 1024, "one block in 100 KB");
  for (const void* f : {(const void*)k_sel_cluster<false>, (const void*)k_sel_cluster<true>})
    ARA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  done[dev] = ctx;
  return ARA_OK;
}

size_t select_scratch_bytes(int64_t n, int32_t n_layers, int32_t n_t, int n_sms) {
  return sel_plan_within(n, n_layers, n_t, n_sms, true, SEL_SCRATCH).bytes;
}

// Plan and stream-ordered scratch of a request; with less memory, fewer rows at a time and shorter lists.
static ara_status take_scratch(int64_t n, int32_t n_layers, int32_t n_t, int n_sms, bool beside, cudaStream_t s,
                               SelPlan* y, void** scratch) {
  *y = sel_plan_within(n, n_layers, n_t, n_sms, beside, SEL_SCRATCH);
  while (true) {
    const cudaError_t e = dmalloc_async(scratch, y->bytes, s);
    if (e == cudaSuccess) return ARA_OK;
    if (e != cudaErrorMemoryAllocation) ARA_TRY(e);
    cudaGetLastError();
    const SelPlan less = sel_plan_within(n, n_layers, n_t, n_sms, beside, y->bytes - y->bytes / 4);
    if (less.bytes >= y->bytes) ARA_TRY(e);
    *y = less;
  }
}

// One group of a request: `rows` rows of `d_ylt`, results to `sc` (counted from the group's first row).
static ara_status launch_group(const double* d_ylt, const SelPlan& y, const SelTargets& tg, int32_t rows,
                               const SelScratch& sc, int want_mean, cudaStream_t s) {
  const int64_t n = y.n;
  if (y.small) {
    int pad = 64;
    while (pad < n) pad <<= 1;
    LaunchScope ls(ARA_K_SELECT, s);
    const auto fn = pad <= 1024 ? k_sel_small<2> : pad <= 2048 ? k_sel_small<4> : k_sel_small<8>;
    fn<<<(unsigned)rows, SEL_THREADS, (size_t)pad * 8, s>>>(d_ylt, (int32_t)n, pad, tg, sc, want_mean);
    ARA_TRY(cudaGetLastError());
    return ARA_OK;
  }
  const int skip = debug_skip_arrival();
  if (y.cluster) {
    for (int32_t l0 = 0; l0 < rows; l0 += 32768) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)y.blocks, (unsigned)std::min<int32_t>(32768, rows - l0));
      cfg.blockDim = dim3(SEL_THREADS);
      cfg.dynamicSmemBytes = SEL_SMEM;
      cfg.stream = s;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)y.blocks;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      LaunchScope ls(ARA_K_SELECT, s);
      const auto fn = y.slices > y.blocks ? k_sel_cluster<true> : k_sel_cluster<false>;
      ARA_TRY(cudaLaunchKernelEx(&cfg, fn, d_ylt, n, l0, (unsigned)y.slices, tg, sc, want_mean, skip));
    }
    return ARA_OK;
  }
  const int32_t per = y.at_once();
  for (int32_t l0 = 0; l0 < rows; l0 += per) {
    const dim3 grid((unsigned)y.blocks, (unsigned)std::min(per, rows - l0));
    uint64_t limit = wait_limit_ns();
    int64_t nn = n;
    SelTargets t2 = tg;
    SelScratch s2 = sc;
    int wm = want_mean, sk = skip;
    void* args[] = {(void*)&d_ylt, &nn, &l0, &t2, &s2, &wm, &limit, &sk};
    LaunchScope ls(ARA_K_SELECT, s);
    ARA_TRY(cudaLaunchCooperativeKernel((const void*)k_sel_grid, grid, dim3(SEL_THREADS), args, (size_t)SEL_SMEM, s));
  }
  return ARA_OK;
}

// Launch the whole selection into `scratch` (laid out by `y`, its first part zero-filled here);
// results land in scratch.out / mean.
ara_status launch_select(const double* d_ylt, const SelPlan& y, const SelTargets& tg, void* scratch,
                         int want_mean, cudaStream_t s, SelScratch* out, uint32_t* ext_err = nullptr,
                         double* user_pml = nullptr, double* user_tvar = nullptr,
                         double* user_mean = nullptr, uint32_t* host_err = nullptr) {
  SelScratch sc = carve(scratch, y);
  if (host_err) sc.err = host_err;
  sc.ext_err = ext_err;
  sc.user_pml = user_pml;
  sc.user_tvar = user_tvar;
  sc.user_mean = user_mean;
  const ara_status ready = sel_prepare_kernels();
  if (ready != ARA_OK) return ready;
  const bool counts = !(y.small || y.cluster);    // class counts in global memory, cleared for every group
  for (int32_t g0 = 0; g0 < y.n_layers; g0 += y.per) {
    // (without counts only the error word needs clearing, and the host's is clear)
    if (g0 == 0 ? counts || !host_err : counts) {
      const size_t z = y.off[g0 == 0 ? 1 : 2];
      ARA_TRY(cudaMemsetAsync((char*)scratch + z, 0, y.zero_end - z, s));
    }
    SelScratch g = sc;
    const int64_t l = g0, lt = l * y.n_t;
    g.state += lt;
    g.out += lt;
    g.mean += l;
    g.gt += lt;
    g.eq += lt;
    if (g.user_pml) g.user_pml += l * tg.n_rp;
    if (g.user_tvar) g.user_tvar += l * (y.n_t - tg.n_rp);
    if (g.user_mean) g.user_mean += l;
    const ara_status st = launch_group(d_ylt + l * y.n, y, tg, std::min(y.per, y.n_layers - g0), g, want_mean, s);
    if (st != ARA_OK) return st;
  }
  *out = sc;
  return ARA_OK;
}

}  // namespace ara

using namespace ara;

namespace ara {

ara_status select_one_rank(const double* d_ylt, int64_t n, int32_t n_layers, int64_t m, int n_sms,
                           cudaStream_t s, SelectResult* out, uint32_t* err) {
  SelTargets tg;
  tg.n_t = 1;
  tg.n_rp = 1;               // the key and its counts, no tail sum
  tg.rank[0] = m;
  SelPlan y;
  void* scratch = nullptr;
  ara_status st = take_scratch(n, n_layers, 1, n_sms, false, s, &y, &scratch);
  if (st != ARA_OK) return st;
  SelScratch sc;
  st = launch_select(d_ylt, y, tg, scratch, 0, s, &sc, err);
  if (st != ARA_OK) {
    cudaFreeAsync(scratch, s);
    return st;
  }
  out->scratch = scratch;
  out->thr_key = &sc.state[0].key;
  out->thr_stride = sizeof(SelState) / sizeof(uint64_t);
  out->gt = sc.gt;
  out->eq = sc.eq;
  return ARA_OK;
}

void free_select_result(SelectResult& r, cudaStream_t s) {
  if (r.scratch) cudaFreeAsync(r.scratch, s);
  r.scratch = nullptr;
}

// The host copy of a request's results (out, mean, err) into the caller's arrays.
static ara_status split_results(const double* out, int32_t n_layers, const SelTargets& tg, double* h_pml,
                                double* h_tvar, double* h_mean) {
  const size_t L = (size_t)n_layers, nt = (size_t)tg.n_t, n_rp = (size_t)tg.n_rp;
  uint32_t timed_out = 0;
  memcpy(&timed_out, out + L * nt + L, sizeof(timed_out));
  if (timed_out) return ARA_ETIMEOUT;
  for (size_t l = 0; l < L; ++l) {
    for (size_t i = 0; i < n_rp; ++i) h_pml[l * n_rp + i] = out[l * nt + i];
    for (size_t i = n_rp; i < nt; ++i) h_tvar[l * (nt - n_rp) + i - n_rp] = out[l * nt + i];
    if (h_mean) h_mean[l] = out[L * nt + l];
  }
  return ARA_OK;
}

ara_status risk_metrics_device(const double* d_ylt, int64_t n_trials, int32_t n_layers,
                               int32_t n_rp, const double* rps, int32_t n_tvar,
                               const double* levels, double* h_pml, double* h_tvar,
                               double* h_mean, cudaStream_t s, bool beside) {
  SelTargets tg;
  if (!d_ylt || n_layers < 1) return ARA_EINVAL;
  if ((n_rp > 0 && !h_pml) || (n_tvar > 0 && !h_tvar)) return ARA_EINVAL;
  if ((uintptr_t)d_ylt & 7) return ARA_EINVAL;
  ara_status st = select_targets(n_trials, n_rp, rps, n_tvar, levels, tg);
  if (st != ARA_OK) return st;
  if (tg.n_t == 0 && !h_mean) return ARA_EINVAL;
  int dev = 0, sms = 0;
  ARA_TRY(cudaGetDevice(&dev));
  ARA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SelPlan y;
  void* scratch = nullptr;
  if ((st = take_scratch(n_trials, n_layers, tg.n_t, sms, beside, s, &y, &scratch)) != ARA_OK) return st;
  SelScratch sc;
  const size_t L = (size_t)n_layers, n_pml = L * n_rp, n_tv = L * n_tvar;
  PinnedSlot slot;
  if (slot.p && (n_pml + n_tv + L + 1) * sizeof(double) <= PinnedSlot::kBytes) {
    // the kernel writes the results straight into the pinned block: no copies, one wait
    double* const r = (double*)slot.p;
    volatile uint32_t* const err = (volatile uint32_t*)(r + n_pml + n_tv + L);
    *err = 0u;
    st = launch_select(d_ylt, y, tg, scratch, h_mean != nullptr, s, &sc, nullptr, n_rp > 0 ? r : nullptr,
                       n_tvar > 0 ? r + n_pml : nullptr, h_mean ? r + n_pml + n_tv : nullptr, (uint32_t*)err);
    cudaFreeAsync(scratch, s);
    if (cudaStreamSynchronize(s) != cudaSuccess && st == ARA_OK) st = ARA_ECUDA;
    if (st != ARA_OK) return st;
    if (*err) return ARA_ETIMEOUT;
    std::copy(r, r + n_pml, h_pml);
    std::copy(r + n_pml, r + n_pml + n_tv, h_tvar);
    if (h_mean) std::copy(r + n_pml + n_tv, r + n_pml + n_tv + L, h_mean);
    return ARA_OK;
  }
  st = launch_select(d_ylt, y, tg, scratch, h_mean != nullptr, s, &sc);
  std::vector<double> out(L * tg.n_t + L + 1);   // metrics, means and the error word
  if (st == ARA_OK &&
      cudaMemcpyAsync(out.data(), sc.out, 8 * (out.size() - 1) + 4, cudaMemcpyDeviceToHost, s) != cudaSuccess)
    st = ARA_ECUDA;
  cudaFreeAsync(scratch, s);
  if (cudaStreamSynchronize(s) != cudaSuccess && st == ARA_OK) st = ARA_ECUDA;
  if (st != ARA_OK) return st;
  return split_results(out.data(), n_layers, tg, h_pml, h_tvar, h_mean);
}

}  // namespace ara

namespace ara {
// ara_risk_metrics_async with caller-owned scratch (the host pipeline keeps one per portfolio), within
// `limit` bytes where a plan fits them: ARA_ERANGE with *need set when scratch_bytes is too small, nothing
// queued.
ara_status risk_metrics_queue(const double* d_ylt, int64_t n_trials, int32_t n_layers, int32_t n_rp,
                              const double* rps, int32_t n_tvar, const double* levels,
                              double* d_pml, double* d_tvar, double* d_mean, uint32_t* d_status,
                              void* scratch, size_t scratch_bytes, size_t limit, size_t* need, cudaStream_t s) {
  SelTargets tg;
  if (!d_ylt || n_layers < 1 || !d_status || !need) return ARA_EINVAL;
  if ((n_rp > 0 && !d_pml) || (n_tvar > 0 && !d_tvar)) return ARA_EINVAL;
  if ((uintptr_t)d_ylt & 7) return ARA_EINVAL;
  ara_status st = select_targets(n_trials, n_rp, rps, n_tvar, levels, tg);
  if (st != ARA_OK) return st;
  if (tg.n_t == 0 && !d_mean) return ARA_EINVAL;
  int dev = 0, sms = 0;
  ARA_TRY(cudaGetDevice(&dev));
  ARA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const SelPlan y = sel_plan_within(n_trials, n_layers, tg.n_t, sms, false, std::min(limit, SEL_SCRATCH));
  *need = y.bytes;
  if (!scratch || scratch_bytes < *need) return ARA_ERANGE;
  SelScratch sc;
  ARA_TRY(cudaMemsetAsync(d_status, 0, sizeof(uint32_t), s));
  return launch_select(d_ylt, y, tg, scratch, d_mean != nullptr, s, &sc, d_status,
                       n_rp > 0 ? d_pml : nullptr, n_tvar > 0 ? d_tvar : nullptr, d_mean);
}
}  // namespace ara

extern "C" ara_status ara_risk_metrics_async(const double* d_ylt, int64_t n_trials,
                                             int32_t n_layers, int32_t n_rp, const double* rps,
                                             int32_t n_tvar, const double* levels, double* d_pml,
                                             double* d_tvar, double* d_mean, uint32_t* d_status,
                                             void* stream) {
  SelTargets tg;
  if (!d_ylt || n_layers < 1 || !d_status) return ARA_EINVAL;
  if ((n_rp > 0 && !d_pml) || (n_tvar > 0 && !d_tvar)) return ARA_EINVAL;
  if ((uintptr_t)d_ylt & 7) return ARA_EINVAL;
  ara_status st = select_targets(n_trials, n_rp, rps, n_tvar, levels, tg);
  if (st != ARA_OK) return st;
  if (tg.n_t == 0 && !d_mean) return ARA_EINVAL;
  static_assert(ARA_DEVICE_TIMEOUT == DERR_TIMEOUT, "device timeout flag");
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0, sms = 0;
  ARA_TRY(cudaGetDevice(&dev));
  ARA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SelPlan y;
  void* scratch = nullptr;
  if ((st = take_scratch(n_trials, n_layers, tg.n_t, sms, false, s, &y, &scratch)) != ARA_OK) return st;
  ara_status r = ARA_OK;
  SelScratch sc;
  if (cudaMemsetAsync(d_status, 0, sizeof(uint32_t), s) != cudaSuccess) r = ARA_ECUDA;
  if (r == ARA_OK)   // the kernel writes the results straight into d_pml / d_tvar / d_mean
    r = launch_select(d_ylt, y, tg, scratch, d_mean != nullptr, s, &sc, d_status,
                      n_rp > 0 ? d_pml : nullptr, n_tvar > 0 ? d_tvar : nullptr, d_mean);
  cudaFreeAsync(scratch, s);
  return r;
}

extern "C" ara_status ara_risk_metrics(const double* d_ylt, int64_t n_trials, int32_t n_layers,
                                       int32_t n_rp, const double* rps, int32_t n_tvar,
                                       const double* levels, double* h_pml, double* h_tvar,
                                       double* h_mean, void* stream) {
  return risk_metrics_device(d_ylt, n_trials, n_layers, n_rp, rps, n_tvar, levels, h_pml, h_tvar,
                             h_mean, (cudaStream_t)stream, false);
}

// ------------------------------------------------------------------------------------------
// Allocation-free variant: the selection scratch lives in a fixed device array of this
// library.  Host code cannot use the array's name as a device address, so every call looks the
// address up on the current device (with that device current).  The lookup is a cheap host
// query; not caching it keeps the address right after anything that tears down and recreates
// the device's primary context (cudaDeviceReset), which reloads the module elsewhere.
// ------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_select_scratch[ARA_STATIC_SELECT_BYTES];

static ara_status static_scratch(void** out) {
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_select_scratch);
  if (e != cudaSuccess || !p) {
    note_cuda_error(e, "cudaGetSymbolAddress(g_select_scratch)", __FILE__, __LINE__);
    return ARA_ECUDA;
  }
  *out = p;
  return ARA_OK;
}

extern "C" ara_status ara_risk_metrics_static(const double* d_ylt, int64_t n_trials,
                                              int32_t n_layers, int32_t n_rp, const double* rps,
                                              int32_t n_tvar, const double* levels, double* h_pml,
                                              double* h_tvar, double* h_mean, void* stream) {
  SelTargets tg;
  if (!d_ylt || n_layers < 1) return ARA_EINVAL;
  if ((n_rp > 0 && !h_pml) || (n_tvar > 0 && !h_tvar)) return ARA_EINVAL;
  if ((uintptr_t)d_ylt & 7) return ARA_EINVAL;
  ara_status st = select_targets(n_trials, n_rp, rps, n_tvar, levels, tg);
  if (st != ARA_OK) return st;
  if (tg.n_t == 0 && !h_mean) return ARA_EINVAL;
  int dev = 0, sms = 0;
  ARA_TRY(cudaGetDevice(&dev));
  ARA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // The request's size is bounded as documented (about 8 KiB per layer and level).
  const size_t lt = (size_t)n_layers * (size_t)tg.n_t;
  size_t need = 0;
  for (size_t part : {8192 * lt, 4 * (size_t)n_layers, (size_t)4, 16 * lt, 8 * lt, 8 * lt, 8 * lt, 8 * lt, 8 * lt,
                      8 * lt, 8 * (size_t)n_layers, 8 * (size_t)n_layers})
    need = (need + 255) / 256 * 256 + part;
  if ((need + 255) / 256 * 256 > ARA_STATIC_SELECT_BYTES) return ARA_ERANGE;
  SelGroups g;
  if (!sel_groups(n_trials, n_layers, tg.n_t, sms, ARA_STATIC_SELECT_BYTES, g)) return ARA_ERANGE;
  void* scratch = nullptr;
  if ((st = static_scratch(&scratch)) != ARA_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<double> out((size_t)g.per * (tg.n_t + 1) + 1);
  for (int32_t l0 = 0; l0 < n_layers && st == ARA_OK; l0 += g.per) {
    const SelPlan& y = n_layers - l0 >= g.per ? g.first : g.last;
    SelScratch sc;
    st = launch_select(d_ylt + (int64_t)l0 * n_trials, y, tg, scratch, h_mean != nullptr, s, &sc);
    cudaError_t e = cudaSuccess;
    if (st == ARA_OK) {
      e = cudaMemcpyAsync(out.data(), sc.out, 8 * (size_t)y.n_layers * (tg.n_t + 1) + 4, cudaMemcpyDeviceToHost, s);
      if (e != cudaSuccess) note_cuda_error(e, "static risk metrics: result copy", __FILE__, __LINE__);
    }
    // Always wait for the stream before returning (and before the array is used again), so that no copy
    // queued here can land anywhere after the call has returned.
    const cudaError_t es = cudaStreamSynchronize(s);
    if (e == cudaSuccess && es != cudaSuccess) {
      note_cuda_error(es, "cudaStreamSynchronize", __FILE__, __LINE__);
      e = es;
    }
    if (st == ARA_OK && e != cudaSuccess) st = ARA_ECUDA;
    if (st == ARA_OK)
      st = split_results(out.data(), y.n_layers, tg, h_pml ? h_pml + (size_t)l0 * n_rp : nullptr,
                         h_tvar ? h_tvar + (size_t)l0 * n_tvar : nullptr, h_mean ? h_mean + l0 : nullptr);
  }
  return st;
}
