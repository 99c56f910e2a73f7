// Batched portfolio: every selected layer of a portfolio in one pass over the YET (the program
// and layer loops of Algorithm 1 folded into one launch).
//
// Preparation, per run (all on the stream, captured in the plan's CUDA graph): the event-major rows
// of the selected layers, (slot, q) per non-zero occurrence loss (ara_rows.cu, which also holds the
// stream over them).  Layers that list their ELTs in ascending order, which is what a portfolio
// usually has, get their rows from the portfolio's event-major records in one kernel.  Any other
// selection takes the general way, which keeps the layer's own order of the ELT sum:
//   1. q_i(e) = round(C(sum_j C(x_j(e); R_j, L_j); OccR_i, OccL_i) * 2^f_i) and the hit bitmap
//      of every selected layer i, in one launch of the single-layer fold kernel (slot i of the
//      fold workspace; only the non-zero q are stored).
//   2. per-event counts of non-zero q, read from the bitmaps, and the exclusive scan of the 16-byte
//      pairs that they take (in place: beyond the row's place).
//   3. the rows, in place or end to end as from the records: slot << 56 | q in slot order (q < 2^55; q is read only where the bitmap
//      bit is set), padded to whole pairs with an entry of the spare slot.  The event's row
//      descriptor holds its first entry and, per request of a merged serving pass (slots are
//      grouped by request), the number of its entries in one byte each (a row has at most 255
//      entries, one per slot), so that a trial covered by some of the requests walks only
//      their part of the row.
// Both ways give the same q bit for bit, and the sums are exact integers, so the results equal
// those of the single-layer path bit for bit.

#include <algorithm>
#include <vector>

#include "ara_device.cuh"

namespace ara {

constexpr int BT_MAX_LAYERS = 255;          // slot fits in 8 bits (255 = no slot)
constexpr int BT_SCAN_BLOCK = 1024;

// ------------------------------------------------------------------------------------------
// 2. per-event counts and their exclusive scan (two levels: block sums, then their scan)
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t warp_tot[BT_SCAN_BLOCK / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    uint32_t t = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    warp_tot[lane] = t;   // inclusive over warps
  }
  __syncthreads();
  const uint32_t before = (w > 0 ? warp_tot[w - 1] : 0) + x - v;
  if (total) *total = warp_tot[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before;
}

// count of event e: the number of selected layers whose bitmap has bit e set (the 32 lanes of a
// warp read the same word of each bitmap)
__device__ __forceinline__ uint32_t bt_count(const uint32_t* __restrict__ bits, int64_t bits_stride,
                                             int32_t n_sel, int64_t e) {
  const uint32_t* b = bits + (e >> 5);
  const int sh = (int)(e & 31);
  uint32_t c = 0;
#pragma unroll 8
  for (int i = 0; i < n_sel; ++i) c += (__ldg(b + (int64_t)i * bits_stride) >> sh) & 1u;
  return c;
}

__global__ void __launch_bounds__(BT_SCAN_BLOCK)
k_bt_scan_blocks(const uint32_t* __restrict__ bits, int64_t bits_stride, int32_t n_sel, int64_t n,
                 uint32_t* __restrict__ ptr, uint32_t* __restrict__ block_sums,
                 uint32_t* __restrict__ entries, uint32_t K) {
  const int64_t e = (int64_t)blockIdx.x * BT_SCAN_BLOCK + threadIdx.x;
  uint32_t v = e < n ? bt_count(bits, bits_stride, n_sel, e) : 0u;
  if (entries) {   // rows in pairs of entries: the scan counts pairs, *entries gets the entries
    __shared__ uint32_t sum;     // one atomic per block (one per warp took 28 us for 2 M events)
    if (threadIdx.x == 0) sum = 0u;
    __syncthreads();
    const uint32_t c = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&sum, c);
    __syncthreads();
    if (threadIdx.x == 0 && sum) atomicAdd(entries, sum);
    v = row_pairs(v, K);
  }
  uint32_t tot;
  const uint32_t ex = block_excl_scan(v, &tot);
  if (e < n) ptr[e] = ex;
  if (threadIdx.x == 0) block_sums[blockIdx.x] = tot;
}

// single block: exclusive scan of the block sums (loops for many blocks)
__global__ void __launch_bounds__(BT_SCAN_BLOCK)
k_bt_scan_sums(uint32_t* __restrict__ block_sums, int64_t n_blocks, uint32_t* __restrict__ total) {
  uint32_t carry = 0;
  for (int64_t b0 = 0; b0 < n_blocks; b0 += BT_SCAN_BLOCK) {
    const int64_t b = b0 + threadIdx.x;
    const uint32_t v = b < n_blocks ? block_sums[b] : 0u;
    uint32_t tot;
    const uint32_t ex = block_excl_scan(v, &tot);
    if (b < n_blocks) block_sums[b] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) *total = carry;
}

__global__ void k_bt_scan_add(uint32_t* __restrict__ ptr, int64_t n, const uint32_t* __restrict__ block_sums,
                              const uint32_t* __restrict__ total) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) ptr[e] += block_sums[e / BT_SCAN_BLOCK];
  if (e == n) ptr[n] = *total;
}

// Row pointers of an event-major table: ptr[e] = number of set bits of event e over all
// n_sel bitmaps before e (exclusive scan), ptr[n] = total; block_sums holds ceil(n / 1024)
// words of scratch, total one word.  With entries set (one zeroed word) the scan counts pairs of bits,
// every event's count rounded up, and *entries gets the number of bits.
ara_status launch_event_scan(const uint32_t* bits, int64_t bits_stride, int32_t n_sel, int64_t n,
                             uint32_t* ptr, uint32_t* block_sums, uint32_t* total, uint32_t* entries,
                             cudaStream_t s) {
  const int64_t n_blocks = (n + BT_SCAN_BLOCK - 1) / BT_SCAN_BLOCK;
  k_bt_scan_blocks<<<(unsigned)n_blocks, BT_SCAN_BLOCK, 0, s>>>(bits, bits_stride, n_sel, n, ptr,
                                                              block_sums, entries, 0u);
  k_bt_scan_sums<<<1, BT_SCAN_BLOCK, 0, s>>>(block_sums, n_blocks, total);
  k_bt_scan_add<<<(unsigned)((n + 1 + 255) / 256), 256, 0, s>>>(ptr, n, block_sums, total);
  ARA_TRY(cudaGetLastError());
  return ARA_OK;
}

// ------------------------------------------------------------------------------------------
// 3. rows: one thread per event, layers in slot order, and the event's row descriptor
// ------------------------------------------------------------------------------------------
// Request boundaries of a merged pass, in slots: request r owns [first[r], first[r + 1]); unused
// requests start at BT_MAX_LAYERS + 1 (past every slot).
struct BtReqSlots {
  int32_t first[BT_MAX_REQ + 1];
};

__device__ __forceinline__ uint32_t bt_req_of_slot(const BtReqSlots& rs, int i) {
  return (uint32_t)(i >= rs.first[1]) + (uint32_t)(i >= rs.first[2]) + (uint32_t)(i >= rs.first[3]);
}

// Event e's entries in slot order, put(slot, entry) each, while more().
template <typename M, typename F>
__device__ __forceinline__ void bt_row(int32_t n_sel, const uint64_t* __restrict__ q, const uint32_t* __restrict__ bits,
                                       int64_t bits_stride, int64_t catalogue, int64_t e, M&& more, F&& put) {
  constexpr int U = 8;   // slots per step: their bitmap words and table entries load together
  const uint32_t* b = bits + (e >> 5);
  const int sh = (int)(e & 31);
  for (int i0 = 0; i0 < n_sel && more(); i0 += U) {
    bool hit[U];
    uint64_t v[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      hit[u] = i0 + u < n_sel && ((__ldg(b + (int64_t)(i0 + u) * bits_stride) >> sh) & 1u);
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = hit[u] ? __ldg(q + (int64_t)(i0 + u) * catalogue + e) : 0ull;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (hit[u]) put(i0 + u, ((uint64_t)(i0 + u) << 56) | v[u]);
  }
}

// End to end.
__global__ void __launch_bounds__(256)
k_bt_fill(int32_t n_sel, const uint64_t* __restrict__ q, const uint32_t* __restrict__ bits,
          int64_t bits_stride, int64_t catalogue, const uint32_t* __restrict__ ptr,
          uint64_t* __restrict__ entries, uint64_t* __restrict__ rows, BtReqSlots rs, int first_shift) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= catalogue) return;
  uint64_t pos = 2ull * ptr[e];
  const uint64_t end = 2ull * ptr[e + 1];
  uint32_t lens = 0;   // entries of request r in byte r (one 8-byte descriptor per occurrence)
  bt_row(n_sel, q, bits, bits_stride, catalogue, e, [&] { return pos < end; }, [&](int i, uint64_t v) {
    if (pos < end) {
      entries[pos] = v;
      lens += 1u << (8 * bt_req_of_slot(rs, i));
    }
    ++pos;
  });
  if (pos < end) entries[pos] = (uint64_t)n_sel << 56;   // padding: adds 0 to the spare slot
  rows[e] = (uint64_t)(ptr[e] << first_shift) | ((uint64_t)lens << 32);
}

// In place (one request): the row at table + K e in the form of k_rows_build, a longer one with a
// continuation in its last place and the rest in ovf.
__global__ void __launch_bounds__(256)
k_bt_fill_place(int32_t n_sel, const uint64_t* __restrict__ q, const uint32_t* __restrict__ bits,
                int64_t bits_stride, int64_t catalogue, const uint32_t* __restrict__ ptr, uint32_t K,
                uint64_t* __restrict__ table, uint64_t* __restrict__ ovf, uint64_t* __restrict__ rows) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= catalogue) return;
  const uint32_t first = ptr[e], room = 2u * (ptr[e + 1] - first);   // entries outside the row's place
  uint64_t* const ov = ovf + 2ull * first;
  uint64_t* const row = table + (int64_t)K * e;
  const uint32_t inl = room ? K - 1u : K;         // entries at most in the place
  const uint64_t spare = (uint64_t)n_sel << 56;
  uint64_t held = 0;                              // first of a 16-byte pair
  auto put = [&](uint32_t i, uint64_t v) {
    if (K == 1u) row[0] = v;
    else if (i & 1u) reinterpret_cast<ulonglong2*>(row)[i >> 1] = make_ulonglong2(held, v);
    else held = v;
  };
  uint32_t n = 0;
  bt_row(n_sel, q, bits, bits_stride, catalogue, e, [&] { return n < inl + room; }, [&](int, uint64_t v) {
    if (n < inl) put(n, v);
    else if (n < inl + room) ov[n - inl] = v;
    ++n;
  });
  if (room) {
    if (n - inl < room) ov[n - inl] = spare;
    put(K - 1u, ((uint64_t)(n - inl) << 56) | RW_CONT | first);
  } else {
    for (uint32_t k = n; k < K; ++k) put(k, spare);
  }
  if (rows) rows[e] = (uint64_t)(K * e) | ((uint64_t)n << 32);
}

}  // namespace ara

// ------------------------------------------------------------------------------------------
// Host: plan = scratch + autotuned schedule + CUDA graph of the whole run
// ------------------------------------------------------------------------------------------
using namespace ara;

struct ara_plan {
  Portfolio* pf = nullptr;
  int64_t n_trials = 0, n_events = 0;
  const int64_t* d_off = nullptr;
  const int32_t* d_ids = nullptr;
  std::vector<int32_t> sel;
  double* d_ylt = nullptr;
  uint8_t* d_reg = nullptr;
  // requests of a merged serving pass (one request otherwise: all trials, d_ylt / d_reg)
  int32_t n_req = 1;
  BtReqSlots rs{{0, BT_MAX_LAYERS + 1, BT_MAX_LAYERS + 1, BT_MAX_LAYERS + 1, BT_MAX_LAYERS + 1}};
  int64_t req_t0[BT_MAX_REQ] = {0, 0, 0, 0}, req_t1[BT_MAX_REQ] = {0, 0, 0, 0};
  double* req_ylt[BT_MAX_REQ] = {nullptr, nullptr, nullptr, nullptr};
  uint8_t* req_reg[BT_MAX_REQ] = {nullptr, nullptr, nullptr, nullptr};
  // Whether a trial may lie outside a request's window (its rows hold the window's trials only).
  bool windowed() const { return n_req > 1 || req_t0[0] != 0 || req_t1[0] != n_trials; }
  // The rows (d_rows: their descriptors), from the event-major records (by_event) or the folds.
  bool by_event = false;
  bool own_tables = false;           // never the folds (see run_batched_async)
  RowTable rt;
  RowSchedule sched;
  ulonglong2* part = nullptr;        // sums between passes (sched.passes > 1)
  uint32_t* d_ptr = nullptr;         // general way: scan scratch
  uint32_t* d_bsum = nullptr;
  uint64_t* d_rows = nullptr;
  uint32_t* d_total = nullptr;       // [2] pairs of entries taken, entries
  unsigned long long* d_queue = nullptr;
  int64_t n_blocks = 0;
  double tuned_ms = 0.0;
  int n_kernels = 0;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};

namespace {

// The plan as one request: every selected layer over every trial, into d_ylt / d_reg.
void single_request(ara_plan& P) {
  P.n_req = 1;
  P.req_t0[0] = 0;
  P.req_t1[0] = P.n_trials;
  P.req_ylt[0] = P.d_ylt;
  P.req_reg[0] = P.d_reg;
}

// Entries in place per event: the rule of the rows, and from the folds up to 2 (launches of plans with ELTs
// in descending order, us, end to end / in place: 50,000 trials x 1,000 over 2 M events, 1 layer 464 / 307, 4
// layers 524 / 407, 8 layers 584 / 506 (2 places); 100,000 trials, 16 layers 1,118 / 1,299 (4 places)).
int plan_k(const ara_plan& P) {
  const int K = rows_k(*P.pf, P.sel);
  return P.by_event || K <= 2 ? K : 0;
}

ara_status bt_prep(ara_plan& P, cudaStream_t s, bool fill, int* n_kernels) {
  Portfolio& pf = *P.pf;
  if (P.by_event) {
    if (n_kernels) *n_kernels = 1;
    return launch_rows_build(pf, P.sel, P.rt, P.rs.first, s);
  }
  const int n_sel = (int)P.sel.size();
  const int64_t C = pf.catalogue;
  FoldOutHost fo;
  fo.q = pf.d_q;                 // slot i at d_q + i * C (workspace of the single-layer runs)
  fo.bits = pf.d_bits;
  fo.q_stride = C;
  fo.bits_stride = pf.bm_words;
  fo.by_slot = 1;
  fo.nonzero_only = 1;
  ara_status st = launch_fold_to(pf, n_sel, P.sel.data(), fo, s, false);
  if (st != ARA_OK) return st;
  ARA_TRY(cudaMemsetAsync(P.d_total, 0, 2 * sizeof(uint32_t), s));
  k_bt_scan_blocks<<<(unsigned)P.n_blocks, BT_SCAN_BLOCK, 0, s>>>(pf.d_bits, pf.bm_words, n_sel, C,
                                                                  P.d_ptr, P.d_bsum, P.d_total + 1,
                                                                  (uint32_t)P.rt.K);
  k_bt_scan_sums<<<1, BT_SCAN_BLOCK, 0, s>>>(P.d_bsum, P.n_blocks, P.d_total);
  k_bt_scan_add<<<(unsigned)((C + 1 + 255) / 256), 256, 0, s>>>(P.d_ptr, C, P.d_bsum, P.d_total);
  int k = 4;
  if (fill) {
    const unsigned blocks = (unsigned)((C + 255) / 256);
    if (P.rt.K > 0)
      k_bt_fill_place<<<blocks, 256, 0, s>>>(n_sel, pf.d_q, pf.d_bits, pf.bm_words, C, P.d_ptr, (uint32_t)P.rt.K,
                                             P.rt.table, P.rt.ovf, P.d_rows);
    else
      k_bt_fill<<<blocks, 256, 0, s>>>(n_sel, pf.d_q, pf.d_bits, pf.bm_words, C, P.d_ptr, P.rt.ovf, P.d_rows, P.rs,
                                       P.rt.first_shift);
    ++k;
  }
  ARA_TRY(cudaGetLastError());
  if (n_kernels) *n_kernels = k;
  return ARA_OK;
}

ara_status bt_stream(ara_plan& P, cudaStream_t s) {
  RowsStream r{};
  r.n_trials = P.n_trials;
  r.offsets = P.d_off;
  r.n_events = P.n_events;
  r.ids = P.d_ids;
  r.catalogue = (uint32_t)P.pf->catalogue;
  r.table = P.rt.table;
  r.ovf = P.rt.ovf;
  r.desc = P.d_rows;
  r.first_shift = P.rt.first_shift;
  r.part = P.part;
  r.ns = (int32_t)P.sel.size();
  r.n_req = P.n_req;
  r.windowed = P.windowed();
  r.layers = P.pf->d_layers;
  r.queue = P.d_queue;
  r.err = P.pf->d_err;
  for (int q = 0; q < BT_MAX_REQ; ++q) {
    r.t0[q] = P.req_t0[q];
    r.t1[q] = P.req_t1[q];
    r.ylt[q] = P.req_ylt[q];
    r.regimes[q] = P.req_reg[q];
  }
  for (int q = 0; q <= BT_MAX_REQ; ++q) r.first[q] = P.rs.first[q];
  for (int i = 0; i < r.ns; ++i) r.layer_of[i] = P.sel[(size_t)i];
  if (!r.ylt[0]) return ARA_EINVAL;
  return launch_rows_stream(*P.pf, r, P.rt.K, P.sched, s);
}

void bt_free(ara_plan* P) {
  if (!P) return;
  if (P->exec) cudaGraphExecDestroy(P->exec);
  if (P->graph) cudaGraphDestroy(P->graph);
  void* ptrs[] = {P->d_ptr, P->d_rows, P->d_bsum, P->d_total, P->d_queue, P->rt.table, P->rt.ovf, P->part};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  delete P;
}

}  // namespace

namespace ara {
namespace {
ara_status run_plan_async(ara_plan& P, cudaStream_t s);
}  // namespace

bool batched_fits(const Portfolio& pf, size_t n_sel) {
  return n_sel <= (size_t)BT_MAX_LAYERS && n_sel <= (size_t)pf.n_layers &&
         (int64_t)n_sel * pf.catalogue < ((int64_t)1 << 32);
}

// The batched path as one asynchronous call (no graph, default schedule): scratch comes from the
// stream-ordered allocator, the table is sized by a host-known bound (every non-zero entry of
// layer i is an event of one of its ELTs), and nothing waits on the host.
ara_status run_batched_async(Portfolio& pf, const YltArgs& a, cudaStream_t s, bool own_tables) {
  ara_plan P;
  P.pf = &pf;
  P.n_trials = a.n_trials;
  P.n_events = a.n_events;
  P.d_off = a.offsets;
  P.d_ids = a.ids;
  P.sel.assign(a.sel, a.sel + a.n_sel);
  P.d_ylt = a.ylt;
  P.d_reg = a.regimes;
  if (a.id_base != 0 || a.row_stride != a.n_trials) return ARA_EINVAL;
  P.own_tables = own_tables;
  single_request(P);
  return run_plan_async(P, s);
}

// Several requests in one pass (serving): every layer of the portfolio, request r owning the
// slots [slot_first[r], slot_first[r + 1]) and the trials [t0[r], t1[r]) of the union range.
ara_status run_batched_group_async(Portfolio& pf, const GroupArgs& g, cudaStream_t s) {
  if (g.n_req < 1 || g.n_req > BT_MAX_REQ || g.n_trials < 1 || !g.offsets) return ARA_EINVAL;
  if (g.slot_first[0] != 0 || g.slot_first[g.n_req] != pf.n_layers) return ARA_EINVAL;
  ara_plan P;
  P.pf = &pf;
  P.n_trials = g.n_trials;
  P.n_events = g.n_events;
  P.d_off = g.offsets;
  P.d_ids = g.ids;
  for (int32_t l = 0; l < pf.n_layers; ++l) P.sel.push_back(l);
  P.n_req = g.n_req;
  for (int r = 0; r < BT_MAX_REQ; ++r) {
    P.rs.first[r + 1] = r < g.n_req ? g.slot_first[r + 1] : BT_MAX_LAYERS + 1;
    if (r >= g.n_req) continue;
    if (g.slot_first[r + 1] <= g.slot_first[r] || g.t0[r] < 0 || g.t1[r] <= g.t0[r] ||
        g.t1[r] > g.n_trials || !g.ylt[r])
      return ARA_EINVAL;
    P.req_t0[r] = g.t0[r];
    P.req_t1[r] = g.t1[r];
    P.req_ylt[r] = g.ylt[r];
    P.req_reg[r] = g.reg[r];
  }
  P.rs.first[0] = 0;
  return run_plan_async(P, s);
}

namespace {
// Rows of the plan sized by host-known bounds (every non-zero entry of layer i is an event of one
// of its ELTs), its scratch from the stream-ordered allocator; nothing waits on the host.
ara_status run_plan_async(ara_plan& P, cudaStream_t s) {
  Portfolio& pf = *P.pf;
  if (!batched_fits(pf, P.sel.size())) return ARA_ERANGE;
  const int64_t C = pf.catalogue;
  P.by_event = rows_usable(pf, P.sel);
  for (int K = P.windowed() ? 0 : plan_k(P);; K = 0) {
    P.rt = RowTable{};
    P.rt.K = K;
    const RowSizes z = rows_sizes(pf, P.sel, K);
    P.rt.first_shift = z.first_shift;
    P.sched = rows_schedule((int)P.sel.size(), P.rt.K, z.likely_bytes, z.likely_entries, P.n_trials, P.n_events);
    P.n_blocks = (C + BT_SCAN_BLOCK - 1) / BT_SCAN_BLOCK;
    size_t off = 0;
    auto take = [&](size_t n) { size_t o = (off + 255) / 256 * 256; off = o + n; return o; };
    const size_t o_rows = P.rt.K == 0 ? take(8 * (size_t)C) : 0;
    const size_t o_tab = P.rt.K > 0 ? take(8 * (size_t)P.rt.K * (size_t)C) : 0;
    const size_t o_tot = take(8), o_q = take(8), o_ovf = take(16 * (size_t)z.pairs);
    const size_t o_ptr = P.by_event ? 0 : take(4 * (size_t)(C + 1));
    const size_t o_bsum = P.by_event ? 0 : take(4 * (size_t)P.n_blocks);
    const size_t o_part = P.sched.passes > 1 ? take(16 * (size_t)P.n_trials * P.sel.size()) : 0;
    char* buf = nullptr;
    if (dmalloc_async((void**)&buf, off, s) != cudaSuccess) {
      cudaGetLastError();
      if (P.own_tables || (!P.by_event && K == 0)) return ARA_ENOMEM;
      P.by_event = false;            // the general way, end to end, needs least
      continue;
    }
    if (P.rt.K == 0) P.d_rows = (uint64_t*)(buf + o_rows);
    else P.rt.table = (uint64_t*)(buf + o_tab);
    P.d_total = (uint32_t*)(buf + o_tot);
    P.d_queue = (unsigned long long*)(buf + o_q);
    P.rt.ovf = (uint64_t*)(buf + o_ovf);
    P.rt.ovf_pairs = (uint32_t)std::min<int64_t>(z.pairs, UINT32_MAX);
    P.rt.counters = P.d_total;
    P.rt.desc = P.d_rows;
    if (!P.by_event) {
      P.d_ptr = (uint32_t*)(buf + o_ptr);
      P.d_bsum = (uint32_t*)(buf + o_bsum);
    }
    if (P.sched.passes > 1) P.part = (ulonglong2*)(buf + o_part);
    ara_status st = ARA_OK;
    {
      LaunchScope ls(ARA_K_BATCHED, s, (P.by_event ? 1 : 5) + P.sched.passes);
      st = bt_prep(P, s, true, nullptr);
      if (st == ARA_OK) st = bt_stream(P, s);
    }
    cudaFreeAsync(buf, s);
    return st;
  }
}
}  // namespace
}  // namespace ara

extern "C" {

ara_status ara_plan_batched(ara_portfolio* pf_, int64_t n_trials, const int64_t* d_off,
                            int64_t n_events, const int32_t* d_ids, int32_t n_sel_in,
                            const int32_t* layer_sel, double* d_ylt, uint8_t* d_reg, int32_t flags,
                            void* stream, ara_plan** out) {
  Portfolio* pf = static_cast<Portfolio*>(pf_);
  if (!out) return ARA_EINVAL;
  *out = nullptr;
  if (!pf || n_trials < 1 || n_events < 0 || !d_off || !d_ylt || (n_events > 0 && !d_ids))
    return ARA_EINVAL;
  if (flags & ~ARA_PLAN_AUTOTUNE) return ARA_EINVAL;
  if (((uintptr_t)d_ids & 3) || ((uintptr_t)d_off & 7) || ((uintptr_t)d_ylt & 7)) return ARA_EINVAL;
  if (pf->catalogue > 0xffffffffll) return ARA_ERANGE;
  ara_plan* P = new (std::nothrow) ara_plan();
  if (!P) return ARA_ENOMEM;
  P->pf = pf;
  P->n_trials = n_trials;
  P->n_events = n_events;
  P->d_off = d_off;
  P->d_ids = d_ids ? d_ids : reinterpret_cast<const int32_t*>(d_off);
  P->d_ylt = d_ylt;
  P->d_reg = d_reg;
  single_request(*P);
  if (n_sel_in == 0 && layer_sel == nullptr) {
    for (int32_t l = 0; l < pf->n_layers; ++l) P->sel.push_back(l);
  } else {
    if (n_sel_in < 0 || !layer_sel) { bt_free(P); return ARA_EINVAL; }
    for (int32_t i = 0; i < n_sel_in; ++i) {
      if (layer_sel[i] < 0 || layer_sel[i] >= pf->n_layers) { bt_free(P); return ARA_EINVAL; }
      P->sel.push_back(layer_sel[i]);
    }
  }
  if (P->sel.empty()) { bt_free(P); return ARA_EINVAL; }
  if (!batched_fits(*pf, P->sel.size())) {
    bt_free(P);
    return ARA_ERANGE;
  }
  DeviceGuard g(pf->device);
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t C = pf->catalogue;
  P->n_blocks = (C + BT_SCAN_BLOCK - 1) / BT_SCAN_BLOCK;
  auto fail = [&](ara_status st) {
    cudaStreamSynchronize(s);
    bt_free(P);
    return st;
  };
  P->by_event = rows_usable(*pf, P->sel);
  P->rt.K = plan_k(*P);
  const RowSizes z = rows_sizes(*pf, P->sel, P->rt.K);
  P->rt.first_shift = z.first_shift;
  if ((P->rt.K > 0 && dmalloc(&P->rt.table, 8 * (size_t)P->rt.K * (size_t)C) != cudaSuccess) ||
      dmalloc(&P->d_rows, 8 * (size_t)C) != cudaSuccess || dmalloc(&P->d_total, 8) != cudaSuccess ||
      dmalloc(&P->d_queue, sizeof(unsigned long long)) != cudaSuccess ||
      (!P->by_event && (dmalloc(&P->d_ptr, 4 * (size_t)(C + 1)) != cudaSuccess ||
                        dmalloc(&P->d_bsum, 4 * (size_t)P->n_blocks) != cudaSuccess)))
    return fail(ARA_ENOMEM);
  P->rt.counters = P->d_total;
  P->rt.desc = P->d_rows;
  // size the table once (a first build has no room and only counts): the counts depend on the
  // portfolio only
  ara_status st = bt_prep(*P, s, false, nullptr);
  if (st != ARA_OK) return fail(st);
  uint32_t total[2] = {0, 0};
  if (cudaMemcpyAsync(total, P->d_total, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return fail(ARA_ECUDA);
  if (dmalloc(&P->rt.ovf, 16 * (size_t)std::max<uint32_t>(total[0], 1)) != cudaSuccess) return fail(ARA_ENOMEM);
  P->rt.ovf_pairs = total[0];
  if ((st = bt_prep(*P, s, true, nullptr)) != ARA_OK) return fail(st);
  const int64_t table_bytes = 8 * C * std::max(P->rt.K, 1) + 16 * (int64_t)total[0];
  P->sched = rows_schedule((int)P->sel.size(), P->rt.K, table_bytes, (double)total[1] / (double)C, n_trials, n_events);
  const size_t part_bytes = 16 * (size_t)n_trials * P->sel.size();
  const bool tune = (flags & ARA_PLAN_AUTOTUNE) != 0;
  // room for the sums between passes: where the rule takes several, or where they are tried
  const bool try_passes = tune && P->rt.K == 0 && table_bytes > RW_PASS_BYTES / 2;
  if ((P->sched.passes > 1 || try_passes) && dmalloc(&P->part, part_bytes) != cudaSuccess) {
    cudaGetLastError();
    P->part = nullptr;
    P->sched.passes = 1;
  }
  // schedule: the fastest of the candidates on these inputs, or the rule's
  if (tune) {
    cudaEvent_t a, b;
    if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) return fail(ARA_ECUDA);
    const RowSchedule rule = P->sched;
    RowSchedule best = rule;
    float best_ms = 1e30f;
    for (int nc : {4, 8, 16, 32})
      for (int passes : {1, 2, 3}) {
        if (nc > 2 * rule.nc || 2 * nc < rule.nc) continue;
        if (nc == 32 && P->rt.K == 0) continue;   // rows end to end have 16 columns at most
        if (passes > 1 && !(try_passes && P->part)) continue;
        P->sched = RowSchedule{nc, passes, 0};
        float ms = 0.f, tot = 0.f;
        for (int rep = 0; rep < 3 && st == ARA_OK; ++rep) {
          cudaEventRecord(a, s);
          st = bt_stream(*P, s);
          cudaEventRecord(b, s);
          if (st == ARA_OK && cudaEventSynchronize(b) != cudaSuccess) st = ARA_ECUDA;
          cudaEventElapsedTime(&ms, a, b);
          if (rep > 0) tot += ms;
        }
        if (st == ARA_ERANGE) { st = ARA_OK; continue; }   // too wide for a block's shared memory
        if (st != ARA_OK) {
          cudaEventDestroy(a);
          cudaEventDestroy(b);
          return fail(st);
        }
        if (tot / 2 < best_ms) { best_ms = tot / 2; best = P->sched; }
      }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    P->sched = best;
    P->tuned_ms = best_ms;
  }
  if (P->sched.passes == 1 && P->part) {
    cudaFree(P->part);
    P->part = nullptr;
  }
  // capture the whole run into a graph on a private stream
  cudaStream_t cs;
  if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return fail(ARA_ECUDA);
  const bool timing_was = timing_suspend();
  bool ok = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
  int nk = 0;
  if (ok) ok = bt_prep(*P, cs, true, &nk) == ARA_OK;
  if (ok) ok = bt_stream(*P, cs) == ARA_OK;
  cudaGraph_t graph = nullptr;
  const bool ended = cudaStreamEndCapture(cs, &graph) == cudaSuccess;
  timing_resume(timing_was);
  cudaStreamDestroy(cs);
  if (!ok || !ended || !graph) {
    if (graph) cudaGraphDestroy(graph);
    cudaGetLastError();
    return fail(ARA_ECUDA);
  }
  P->graph = graph;
  P->n_kernels = nk + P->sched.passes;
  if (cudaGraphInstantiate(&P->exec, graph, 0) != cudaSuccess) return fail(ARA_ECUDA);
  if (cudaStreamSynchronize(s) != cudaSuccess) return fail(ARA_ECUDA);
  *out = P;
  return ARA_OK;
}

ara_status ara_run_ylt_requests(ara_portfolio* pf_, int64_t n_trials, const int64_t* d_off,
                                int64_t n_events, const int32_t* d_ids, int32_t n_req,
                                const int32_t* req_layer_first, const int64_t* req_trial_begin,
                                const int64_t* req_trial_end, double* const* d_ylt,
                                uint8_t* const* d_regimes, void* stream) {
  Portfolio* pf = static_cast<Portfolio*>(pf_);
  if (!pf || n_trials < 1 || n_events < 0 || !d_off || (n_events > 0 && !d_ids)) return ARA_EINVAL;
  if (n_req < 1 || !req_layer_first || !req_trial_begin || !req_trial_end || !d_ylt) return ARA_EINVAL;
  if (n_req > BT_MAX_REQ || pf->n_layers > BT_MAX_LAYERS) return ARA_ERANGE;
  if (((uintptr_t)d_ids & 3) || ((uintptr_t)d_off & 7)) return ARA_EINVAL;
  if (pf->catalogue > 0xffffffffll) return ARA_ERANGE;
  GroupArgs g;
  g.n_trials = n_trials;
  g.offsets = d_off;
  g.n_events = n_events;
  g.ids = d_ids ? d_ids : reinterpret_cast<const int32_t*>(d_off);
  g.n_req = n_req;
  if (req_layer_first[0] != 0 || req_layer_first[n_req] != pf->n_layers) return ARA_EINVAL;
  for (int32_t r = 0; r < n_req; ++r) {
    if (req_layer_first[r + 1] <= req_layer_first[r]) return ARA_EINVAL;
    if (req_trial_begin[r] < 0 || req_trial_end[r] <= req_trial_begin[r] || req_trial_end[r] > n_trials)
      return ARA_EINVAL;
    if (!d_ylt[r] || ((uintptr_t)d_ylt[r] & 7)) return ARA_EINVAL;
    g.slot_first[r] = req_layer_first[r];
    g.t0[r] = req_trial_begin[r];
    g.t1[r] = req_trial_end[r];
    g.ylt[r] = d_ylt[r];
    g.reg[r] = d_regimes ? d_regimes[r] : nullptr;
  }
  g.slot_first[n_req] = req_layer_first[n_req];
  DeviceGuard dg(pf->device);
  return run_batched_group_async(*pf, g, (cudaStream_t)stream);
}

ara_status ara_plan_launch(ara_plan* P, void* stream) {
  if (!P || !P->exec) return ARA_EINVAL;
  DeviceGuard g(P->pf->device);
  cudaStream_t s = (cudaStream_t)stream;
  LaunchScope ls(ARA_K_BATCHED, s, P->n_kernels);
  ARA_TRY(cudaGraphLaunch(P->exec, s));
  return ARA_OK;
}

ara_status ara_plan_info(ara_plan* P, int32_t* warps, int32_t* bpsm, int32_t* tpg, double* ms,
                         int32_t* copies) {
  if (!P) return ARA_EINVAL;
  if (warps) *warps = RW_WARPS;
  if (bpsm) *bpsm = P->sched.blocks;
  if (tpg) *tpg = 1;
  if (ms) *ms = P->tuned_ms;
  if (copies) *copies = std::min(P->sched.nc, 4);
  return ARA_OK;
}

ara_status ara_plan_table(ara_plan* P, const uint64_t** d_rows, int64_t* n_entries) {
  if (!P || !P->d_rows || !P->d_total) return ARA_EINVAL;
  DeviceGuard g(P->pf->device);
  if (d_rows) *d_rows = P->d_rows;
  if (n_entries) {
    uint32_t total = 0;
    ARA_TRY(cudaDeviceSynchronize());
    ARA_TRY(cudaMemcpy(&total, P->d_total + 1, 4, cudaMemcpyDeviceToHost));
    *n_entries = total;
  }
  return ARA_OK;
}

void ara_plan_destroy(ara_plan* P) {
  if (!P) return;
  DeviceGuard g(P->pf->device);
  cudaDeviceSynchronize();
  bt_free(P);
}

}  // extern "C"
