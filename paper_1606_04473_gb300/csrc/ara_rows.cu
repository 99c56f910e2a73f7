// Event-major rows: every selected layer's non-zero occurrence losses of one catalogue event side
// by side, and the stream of the YET over them (several layers in one pass, Algorithm 1's layer
// loop folded into Algorithm 3's event loop).
//
//   1. k_ev_index (once per portfolio): the ELT records again, event by event (Eq. 2 transposed):
//      the records of event e are [ptr[e], ptr[e + 1]), ELTs ascending.
//   2. k_rows_build (every run): one thread per event walks its records, applies the ELT terms,
//      adds each to the sums of the layers that hold the ELT (ELTs ascending: the order of the
//      per-layer fold when a layer lists its ELTs in ascending order, which is required), applies
//      the occurrence terms and writes the non-zero q, tagged with their slots, as the event's row.
//   3. k_rows_stream (every run): reads every occurrence once, fetches its event's row and adds
//      the entries to the trial's sums; aggregate terms at the end of the trial.
//
// A row has a fixed place and size (K entries of 8 bytes at table + K e, K a power of two chosen
// near the average row length), so an occurrence costs one aligned gather that depends on nothing
// but its ID.  An entry is slot << 56 | q with q < 2^55; spare entries name the slot ns (a sum that
// nobody reads) with q = 0.  A longer row keeps K - 1 entries and, in its last place, a
// continuation (bit 55 set): the first 16-byte pair and the number of further entries in the
// overflow list.  Integer sums make the result independent of the order of the additions.

#include <algorithm>
#include <cmath>
#include <vector>

#include "ara_device.cuh"

namespace ara {

// Non-returning 64-bit shared-memory add.
__device__ __forceinline__ void red_u64(unsigned long long* a, unsigned long long q) {
  asm volatile("red.shared.add.u64 [%0], %1;" :: "r"((uint32_t)__cvta_generic_to_shared(a)), "l"(q) : "memory");
}
constexpr uint64_t RW_Q = (1ull << 55) - 1;

// ------------------------------------------------------------------------------------------
// 1. Event-major records of the portfolio
// ------------------------------------------------------------------------------------------
constexpr int EV_THREADS = 256;
constexpr int EV_GROUP = 32;                      // ELTs whose records are placed together

// One block per fold tile.  The tile's first record in the event-major order is the number of
// records of all ELTs before the tile.  Counts per event, their block scan, then the records in
// groups of 32 ELTs: within a group a record's place among its event's is the number of smaller
// ELTs of the group that hold the event (a 32-bit mask per event), so the order is by ELT.
template <typename LossT>
__global__ void __launch_bounds__(EV_THREADS)
k_ev_index(int64_t catalogue, int32_t n_elts, const int64_t* __restrict__ rec_off,
           const int64_t* __restrict__ tile_rec, int64_t n_tiles, const int32_t* __restrict__ rec_ids,
           const LossT* __restrict__ rec_loss, uint32_t* __restrict__ ptr, int32_t* __restrict__ ev_elt,
           LossT* __restrict__ ev_loss) {
  __shared__ uint32_t cur[FOLD_TILE];
  __shared__ uint32_t mask[FOLD_TILE];
  __shared__ int64_t lo[EV_GROUP];
  __shared__ int32_t off[EV_GROUP + 1];
  __shared__ unsigned long long base_s;
  __shared__ uint32_t part[EV_THREADS];
  const int64_t b = blockIdx.x, t0 = b * FOLD_TILE;
  for (int i = threadIdx.x; i < FOLD_TILE; i += EV_THREADS) cur[i] = mask[i] = 0u;
  if (threadIdx.x == 0) base_s = 0ull;
  __syncthreads();
  unsigned long long mine = 0;
  for (int32_t j = threadIdx.x; j < n_elts; j += EV_THREADS)
    mine += (unsigned long long)(tile_rec[(int64_t)j * (n_tiles + 1) + b] - rec_off[j]);
  if (mine) atomicAdd(&base_s, mine);
  // the group's record ranges in this tile; every thread gets the group's record count
  auto load_group = [&](int32_t j0) -> int32_t {
    __syncthreads();
    if (threadIdx.x < 32) {
      const int32_t j = j0 + (int32_t)threadIdx.x;
      int32_t c = 0;
      if (j < n_elts) {
        const int64_t* tr = tile_rec + (int64_t)j * (n_tiles + 1) + b;
        lo[threadIdx.x] = tr[0];
        c = (int32_t)(tr[1] - tr[0]);
      }
      int32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t v = __shfl_up_sync(FULL, incl, o);
        if ((int)threadIdx.x >= o) incl += v;
      }
      off[threadIdx.x + 1] = incl;
      if (threadIdx.x == 0) off[0] = 0;
    }
    __syncthreads();
    return off[EV_GROUP];
  };
  auto find = [&](int32_t x) -> int {   // the group's ELT that owns record x
    int g = 0;
#pragma unroll
    for (int step = EV_GROUP / 2; step > 0; step >>= 1)
      if (off[g + step] <= x) g += step;
    return g;
  };
  for (int32_t j0 = 0; j0 < n_elts; j0 += EV_GROUP) {
    const int32_t n = load_group(j0);
    for (int32_t x = threadIdx.x; x < n; x += EV_THREADS) {
      const int g = find(x);
      atomicAdd(&cur[(int)(rec_ids[lo[g] + (x - off[g])] - t0)], 1u);
    }
  }
  __syncthreads();
  {   // exclusive scan of the counts; cur becomes the next free place of every event
    constexpr int PER = FOLD_TILE / EV_THREADS;
    uint32_t s = 0;
    for (int i = 0; i < PER; ++i) s += cur[threadIdx.x * PER + i];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < EV_THREADS; o <<= 1) {
      const uint32_t v = (int)threadIdx.x >= o ? part[threadIdx.x - o] : 0u;
      __syncthreads();
      part[threadIdx.x] += v;
      __syncthreads();
    }
    uint32_t run = (uint32_t)base_s + part[threadIdx.x] - s;
    for (int i = 0; i < PER; ++i) {
      const int e = threadIdx.x * PER + i;
      const uint32_t c = cur[e];
      cur[e] = run;
      if (t0 + e <= catalogue) ptr[t0 + e] = run;
      run += c;
    }
    // the last tile ends on the catalogue: its end has no thread of its own
    if (t0 + FOLD_TILE == catalogue && threadIdx.x == EV_THREADS - 1) ptr[catalogue] = run;
  }
  for (int32_t j0 = 0; j0 < n_elts; j0 += EV_GROUP) {
    const int32_t n = load_group(j0);
    if (n == 0) continue;                         // uniform over the block
    for (int32_t x = threadIdx.x; x < n; x += EV_THREADS) {
      const int g = find(x);
      atomicOr(&mask[(int)(rec_ids[lo[g] + (x - off[g])] - t0)], 1u << g);
    }
    __syncthreads();
    for (int32_t x = threadIdx.x; x < n; x += EV_THREADS) {
      const int g = find(x);
      const int64_t r = lo[g] + (x - off[g]);
      const int e = (int)(rec_ids[r] - t0);
      const uint32_t at = cur[e] + __popc(mask[e] & ((1u << g) - 1u));
      ev_elt[at] = j0 + g;
      ev_loss[at] = rec_loss[r];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < FOLD_TILE; i += EV_THREADS) {
      cur[i] += __popc(mask[i]);
      mask[i] = 0u;
    }
  }
}

// Builds the portfolio's event-major records.  Best effort: without room for them the portfolio
// works through the per-layer folds alone.
ara_status build_event_index(Portfolio& pf, cudaStream_t s) {
  if (pf.n_records < 1 || pf.n_records >= (int64_t)UINT32_MAX || pf.catalogue > RW_MAX_CATALOGUE) return ARA_OK;
  const size_t esz = pf.d_rec_loss32 ? sizeof(float) : sizeof(double);
  const size_t o_elt = ((size_t)(pf.catalogue + 1) * 4 + 255) / 256 * 256;
  const size_t o_loss = o_elt + ((size_t)pf.n_records * 4 + 255) / 256 * 256;
  char* buf = nullptr;
  if (dmalloc(&buf, o_loss + (size_t)pf.n_records * esz) != cudaSuccess) {
    cudaGetLastError();
    return ARA_OK;
  }
  pf.d_ev_ptr = (uint32_t*)buf;
  pf.d_ev_elt = (int32_t*)(buf + o_elt);
  pf.d_ev_loss = buf + o_loss;
  LaunchScope ls(ARA_K_FOLD, s);
  if (pf.d_rec_loss32)
    k_ev_index<float><<<(unsigned)pf.n_tiles, EV_THREADS, 0, s>>>(
        pf.catalogue, pf.n_elts, pf.d_rec_off, pf.d_tile_rec, pf.n_tiles, pf.d_rec_ids, pf.d_rec_loss32,
        pf.d_ev_ptr, pf.d_ev_elt, (float*)pf.d_ev_loss);
  else
    k_ev_index<double><<<(unsigned)pf.n_tiles, EV_THREADS, 0, s>>>(
        pf.catalogue, pf.n_elts, pf.d_rec_off, pf.d_tile_rec, pf.n_tiles, pf.d_rec_ids, pf.d_rec_loss,
        pf.d_ev_ptr, pf.d_ev_elt, (double*)pf.d_ev_loss);
  ARA_TRY(cudaGetLastError());
  return ARA_OK;
}

// ------------------------------------------------------------------------------------------
// 2. Rows
// ------------------------------------------------------------------------------------------
struct RowsBuild {
  int64_t catalogue;
  const uint32_t* ptr;
  const int32_t* elt;
  const void* loss;
  const double* elt_ret;
  const double* elt_lim;
  const uint64_t* mem;         // [n_elts][RW_MASK]: bit l set when layer l holds the ELT
  const LayerConst* layers;
  int32_t n_layers;
  int32_t ns;
  int32_t K;
  uint64_t* table;
  uint64_t* ovf;
  uint32_t ovf_pairs;          // capacity of ovf in 16-byte pairs (0: only count)
  uint32_t* counters;          // [0] overflow pairs taken, [1] entries in all rows
  uint64_t* desc;              // [catalogue]: first entry | number of entries << 32 (optional, K > 0)
  // ADJ only: entries are slots (one byte) of the layers whose occurrence regime is not 0, K = 0, and a
  // descriptor holds the first slots too (ara_adjoint.cu)
  uint8_t* ent;
  uint8_t* regime;             // [ns][catalogue], zeroed
  AdjbSlots q;
  int32_t first_shift;
  int32_t first[5];            // first slot of each request (as RowsStream)
  uint64_t sel[RW_MASK];       // the selected layers
  uint8_t slot_of[256];        // layer -> slot
};

struct RowsLayer {             // staged per block
  double occ_ret, occ_lim;
  int32_t frac_bits, slot;
};

// Exclusive block scan of v; *total gets the sum.
__device__ __forceinline__ uint32_t rb_scan(uint32_t v, uint32_t* part, uint32_t* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31) part[wid] = incl;
  __syncthreads();
  uint32_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < RW_BUILD_THREADS / 32; ++w) {
    const uint32_t x = part[w];
    if (w < wid) before += x;
    all += x;
  }
  __syncthreads();
  *total = all;
  return before + incl - v;
}

// One thread per event.  The bit masks of its ELTs' layers tell which layers it can reach; their
// sums lie side by side in shared memory, packed over the block's events (a sum's place is its
// layer's rank in the event's mask), so that a block holds little and many run at once: the walk
// is a chain of dependent loads.  A first term is stored, not added (0 + x = x): FP64 instructions
// issue at 2 lanes per clock and SM here, whatever the number of active lanes.  Events whose sums
// do not fit take another turn.
template <typename LossT, int MW, bool ADJ>
__global__ void __launch_bounds__(RW_BUILD_THREADS)
k_rows_build(RowsBuild p) {
  __shared__ double acc[RW_BUILD_SUMS];
  __shared__ uint32_t part[RW_BUILD_THREADS / 32];
  __shared__ uint32_t base_s;
  extern __shared__ __align__(16) unsigned char rb_smem[];
  RowsLayer* const lay = reinterpret_cast<RowsLayer*>(rb_smem);   // [n_layers]
  const int tid = threadIdx.x;
  for (int i = tid; i < p.n_layers; i += RW_BUILD_THREADS) {
    const LayerConst& lc = p.layers[i];
    lay[i] = RowsLayer{lc.occ_ret, lc.occ_lim, lc.frac_bits, (int)p.slot_of[i]};
  }
  const int64_t e = (int64_t)blockIdx.x * RW_BUILD_THREADS + tid;
  const LossT* const loss = reinterpret_cast<const LossT*>(p.loss);
  uint32_t r0 = 0, r1 = 0;
  if (e < p.catalogue) {
    r0 = __ldg(p.ptr + e);
    r1 = __ldg(p.ptr + e + 1);
  }
  uint64_t reach[MW];
#pragma unroll
  for (int w = 0; w < MW; ++w) reach[w] = 0ull;
  for (uint32_t r = r0; r < r1; ++r) {
    const uint64_t* const m = p.mem + (int64_t)__ldg(p.elt + r) * RW_MASK;
#pragma unroll
    for (int w = 0; w < MW; ++w) reach[w] |= __ldg(m + w);
  }
  uint32_t n_reach = 0, before[MW];               // sums of the words below each word
#pragma unroll
  for (int w = 0; w < MW; ++w) {
    reach[w] &= p.sel[w];
    before[w] = n_reach;
    n_reach += (uint32_t)__popcll(reach[w]);
  }
  uint32_t total;
  const uint32_t place = rb_scan(n_reach, part, &total);
  uint32_t lo = 0;                                // first sum of this turn
  bool todo = e < p.catalogue;
  while (true) {
    const bool mine = todo && place + n_reach - lo <= (uint32_t)RW_BUILD_SUMS;
    double* const x = acc + (mine ? place - lo : 0u);
    uint64_t begun[MW];
#pragma unroll
    for (int w = 0; w < MW; ++w) begun[w] = 0ull;
    uint32_t n = 0;
    if (mine) {
      for (uint32_t r = r0; r < r1; ++r) {
        const int j = __ldg(p.elt + r);
        const double a = clamp_terms_bits(to_f64(__ldg(loss + r)), __ldg(p.elt_ret + j), __ldg(p.elt_lim + j));
        if (((uint64_t)__double_as_longlong(a) << 1) == 0ull) continue;
#pragma unroll
        for (int w = 0; w < MW; ++w)
          for (uint64_t m = __ldg(p.mem + (int64_t)j * RW_MASK + w) & p.sel[w]; m; m &= m - 1) {
            const uint64_t bit = m & (0ull - m);
            double* const s = x + before[w] + __popcll(reach[w] & (bit - 1));
            double v = a;
            if (begun[w] & bit) v = __dadd_rn(*s, a);
            *s = v;
            begun[w] |= bit;
          }
      }
      // occurrence terms; layers whose q is 0 leave the mask
#pragma unroll
      for (int w = 0; w < MW; ++w)
        for (uint64_t m = begun[w]; m; m &= m - 1) {
          const uint64_t bit = m & (0ull - m);
          const RowsLayer& l = lay[64 * w + __ffsll((long long)m) - 1];
          double* const s = x + before[w] + __popcll(reach[w] & (bit - 1));
          uint64_t q;
          if (ADJ) {   // the regime: inside the cover or above it
            const long long ex = __double_as_longlong(__dsub_rn(*s, l.occ_ret));
            const long long lim = __double_as_longlong(l.occ_lim);
            q = ex > 0 ? (ex < lim ? 1ull : ex > lim ? 2ull : 0ull) : 0ull;
          } else {
            q = fixed_rn(clamp_terms_bits(*s, l.occ_ret, l.occ_lim), l.frac_bits);
          }
          if (q) {
            *s = __longlong_as_double((long long)q);
            ++n;
          } else {
            begun[w] ^= bit;
          }
        }
    }
    // room for the rows (K = 0) or their overflow, one atomic per block
    const uint32_t more = p.K == 0 ? n : n > (uint32_t)p.K ? n - (uint32_t)p.K + 1u : 0u;
    const uint32_t need = row_pairs(n, (uint32_t)p.K);
    uint32_t pairs, cnt;
    uint32_t at = rb_scan(need, part, &pairs);
    rb_scan(n, part, &cnt);
    if (tid == 0) {
      base_s = pairs ? atomicAdd(p.counters, pairs) : 0u;
      if (cnt) atomicAdd(p.counters + 1, cnt);
    }
    __syncthreads();
    at += base_s;                                 // first pair of this row's part of ovf
    if (ADJ && mine && at + need <= p.ovf_pairs) {
      uint64_t desc = 2ull * at | ((uint64_t)n << 32);
      uint32_t k = 0;
#pragma unroll
      for (int w = 0; w < MW; ++w)
        for (uint64_t m = begun[w]; m; m &= m - 1) {
          const uint64_t bit = m & (0ull - m);
          const int s = lay[64 * w + __ffsll((long long)m) - 1].slot;
          const double r = x[before[w] + __popcll(reach[w] & (bit - 1))];
          p.regime[(int64_t)s * p.catalogue + e] = (uint8_t)__double_as_longlong(r);
          p.ent[2 * (int64_t)at + k] = (uint8_t)s;
          if (k < p.q.n) desc |= (uint64_t)s << (40u + p.q.width * k);
          ++k;
        }
      p.desc[e] = desc;
    }
    if (!ADJ && mine && !(need && at + need > p.ovf_pairs)) {   // else a counting run
      const uint64_t spare = (uint64_t)p.ns << 56;
      uint64_t* const ov = p.ovf + 2 * (int64_t)at;
      uint64_t* const row = p.table + (int64_t)p.K * e;
      const uint32_t inl = p.K == 0 ? 0u : more ? (uint32_t)p.K - 1u : n;   // entries kept in the row
      uint32_t k = 0, lens = 0;
      uint64_t held = 0;                          // first of a 16-byte pair
      auto put = [&](uint32_t i, uint64_t v) {    // entry i of the row, in order
        if (p.K == 1) row[0] = v;
        else if (i & 1u) reinterpret_cast<ulonglong2*>(row)[i >> 1] = make_ulonglong2(held, v);
        else held = v;
      };
#pragma unroll
      for (int w = 0; w < MW; ++w)
        for (uint64_t m = begun[w]; m; m &= m - 1) {
          const uint64_t bit = m & (0ull - m);
          const int s = lay[64 * w + __ffsll((long long)m) - 1].slot;
          const uint64_t q = (uint64_t)__double_as_longlong(x[before[w] + __popcll(reach[w] & (bit - 1))]);
          const uint64_t v = ((uint64_t)s << 56) | q;
          if (k < inl) put(k, v);
          else ov[k - inl] = v;
          ++k;
          lens += 1u << (8 * ((s >= p.first[1]) + (s >= p.first[2]) + (s >= p.first[3])));
        }
      if (more & 1u) ov[more] = spare;
      if (p.K == 0) {
        p.desc[e] = (uint64_t)(at << p.first_shift) | ((uint64_t)lens << 32);
      } else {
        if (more) put((uint32_t)p.K - 1u, ((uint64_t)more << 56) | RW_CONT | (uint64_t)at);
        else
          for (; k < (uint32_t)p.K; ++k) put(k, spare);
        if (p.desc) p.desc[e] = (uint64_t)(p.K * e) | ((uint64_t)n << 32);
      }
    }
    if (mine) todo = false;
    if (total - lo <= (uint32_t)RW_BUILD_SUMS) return;     // uniform: the last turn
    // next turn: from the first event left (places ascend with the thread index)
    __syncthreads();
    if (tid == 0) base_s = total;
    __syncthreads();
    if (todo) atomicMin(&base_s, place);
    __syncthreads();
    lo = base_s;
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// 3. Stream
// ------------------------------------------------------------------------------------------
constexpr int RW_U = 2;                // windows of 32 pairs in flight together
constexpr int RW_SEG_ROUNDS = 14;      // rounds of 32 occurrences between two drains (see below)
constexpr int RW_PEND = 64;            // rows whose continuation waits to be walked

// Adds of a segment: at most one value below 2^55 per occurrence and slot, over at most 14 rounds
// of 32 occurrences and 32 waiting continuations: 480 values, whose sum stays below 2^64.
static_assert(RW_SEG_ROUNDS * 32 + 32 <= 512, "a 64-bit column must not wrap");

// Adds two entries of a row to the lane's column (a != b, or both add 0: a row holds a slot once).
// Lanes that share a column take turns with plain loads and stores; with 4 columns eight turns cost
// more than the atomics they replace (64 layers: 6.0 against 5.0 ms; with 8 columns 4.27 against 4.6).
template <int NC>
__device__ __forceinline__ void add_columns(unsigned long long* a, unsigned long long* b,
                                            unsigned long long qa, unsigned long long qb, int lane) {
  if constexpr (NC == 4) {
    red_u64(a, qa);
    red_u64(b, qb);
  } else {
    constexpr int PH = 32 / NC;
#pragma unroll
    for (int ph = 0; ph < PH; ++ph) {
      if (PH == 1 || lane / NC == ph) {
        const unsigned long long sa = *a, sb = *b;
        *a = sa + qa;
        *b = sb + qb;
      }
      if (PH > 1) __syncwarp();
    }
  }
}

// Lanes of a warp take the rows of 32 occurrences (a round) LPR = K / 2 lanes to a row, 16 bytes
// each, RPW rows at a time.  Each lane adds its entries to a column of 64-bit sums of its own
// (NC = 32 columns) or shared by 32 / NC lanes that take turns: plain loads and stores, the lanes
// of a turn in different banks whatever their slots.  Continuations are collected and walked 32
// rows at a time as one joined list of pairs.
template <int K, int NC>
__global__ void __launch_bounds__(RW_WARPS * 32, RW_MIN_BLOCKS)
k_rows_stream(RowsStream p) {
  constexpr int LPR = K >= 2 ? K / 2 : 1, RPW = 32 / LPR;
  constexpr int B = LPR < 4 ? LPR : 4;            // windows of RPW rows in flight together
  constexpr int NB = LPR / B;                     // batches of B windows per round
  constexpr int PH = 32 / NC;
  constexpr uint32_t NONE = 0xffffffffu;
  extern __shared__ __align__(16) unsigned long long rw_smem[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ns = p.ns;
  const uint32_t lt = (1u << lane) - 1u, le = lt | (1u << lane);
  // per warp: [ns + 1][NC] columns, [2][ns] totals, the waiting rows (pair, pairs), 32 row bases
  const int words = (ns + 1) * NC + 2 * ns + RW_PEND + 16;
  unsigned long long* const acc0 = rw_smem + (int64_t)wid * words;
  unsigned long long* const tot = acc0 + (ns + 1) * NC;
  unsigned long long* const pend = tot + 2 * ns;
  uint32_t* const rbase = reinterpret_cast<uint32_t*>(pend + RW_PEND);
  unsigned long long* const col = acc0 + (lane & (NC - 1));
  const int rot = NC >= 16 ? lane : (NC == 8 ? lane >> 1 : lane >> 2);
  for (int i = lane; i < words; i += 32) acc0[i] = 0ull;
  __syncwarp();
  bool bad_id = false, bad_off = false;

  auto grab = [&]() -> unsigned long long {       // lane 0's value; broadcast where it is used
    return lane == 0 ? atomicAdd(p.queue, 1ull) : 0ull;
  };
  auto add_pair = [&](const ulonglong2& v) {
    unsigned long long* const a = col + (uint32_t)(v.x >> 56) * NC;
    unsigned long long* const b = col + (uint32_t)(v.y >> 56) * NC;
    const unsigned long long qa = v.x & RW_Q, qb = v.y & RW_Q;
    add_columns<NC>(a, b, qa, qb, lane);
  };
  auto add_one = [&](uint64_t v) {
    unsigned long long* const a = col + (uint32_t)(v >> 56) * NC;
    if constexpr (NC == 4) {
      red_u64(a, v & RW_Q);
    } else {
#pragma unroll
      for (int ph = 0; ph < PH; ++ph) {
        if (PH == 1 || lane / NC == ph) *a += v & RW_Q;
        if (PH > 1) __syncwarp();
      }
    }
  };
  int np = 0;                                     // waiting continuations
  auto walk = [&](int cnt) {                      // the first cnt (<= 32) of them
    const uint64_t w = lane < cnt ? pend[lane] : 0ull;
    const uint32_t nch = (uint32_t)(w >> 32);
    uint32_t incl = nch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += v;
    }
    const uint32_t total = __shfl_sync(FULL, incl, 31), excl = incl - nch;
    if (nch) rbase[lane] = (uint32_t)w - excl;    // every waiting row has a pair: rank = lane
    const uint64_t keep = lane + cnt < np ? pend[lane + cnt] : 0ull;
    __syncwarp();
    int started = -1;
    for (uint32_t w0 = 0; w0 < total; w0 += 32) {
      const uint32_t rel = excl - w0;
      const uint32_t m = __reduce_or_sync(FULL, (nch != 0u && rel < 32u) ? 1u << rel : 0u);
      const int own = started + __popc(m & le);
      started += __popc(m);
      const uint32_t x = w0 + (uint32_t)lane;
      ulonglong2 v = make_ulonglong2(0ull, 0ull);
      if (x < total) v = __ldcg(reinterpret_cast<const ulonglong2*>(p.ovf) + (uint32_t)(rbase[own] + x));
      add_pair(v);
    }
    __syncwarp();
    np -= cnt;
    if (lane < np) pend[lane] = keep;             // at most 32 stay
    __syncwarp();
  };
  auto push = [&](bool c, uint64_t v) {           // continuations of one window
    const uint32_t m = __ballot_sync(FULL, c);
    if (m == 0u) return;
    if (c) pend[np + __popc(m & lt)] = (((v >> 57) + ((v >> 56) & 1ull)) << 32) | (uint32_t)v;
    np += __popc(m);
    __syncwarp();
    if (np > 32) walk(32);
  };
  auto drain = [&](int i) -> U128 {               // slot i: its total and columns, cleared
    U128 S{tot[i], tot[ns + i]};
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      unsigned long long* const a = acc0 + i * NC + ((c + rot) & (NC - 1));
      add_u64(S, *a);
      *a = 0ull;
    }
    return S;
  };

  unsigned long long g_next = 0;
  int64_t t = (int64_t)__shfl_sync(FULL, grab(), 0);
  g_next = grab();
  int64_t beg = 0, end = 0;
  auto load_id = [&](int64_t i) -> uint32_t {     // NONE past the trial's end and for a bad ID
    if (i >= end) return NONE;
    const uint32_t e = (uint32_t)__ldcs(p.ids + i);
    if (e < p.catalogue) return e;
    bad_id = true;
    return NONE;
  };
  auto check_range = [&]() {
    if (!(0 <= beg && beg <= end && end <= p.n_events)) { bad_off = true; beg = end = 0; }
  };
  uint32_t e_cur = NONE, e_nxt = NONE;
  if (t < p.n_trials) {
    beg = __ldg(p.offsets + t);
    end = __ldg(p.offsets + t + 1);
    check_range();
    e_cur = load_id(beg + lane);
    e_nxt = load_id(beg + 32 + lane);
  }
  while (t < p.n_trials) {
    // the next trial's place in the queue is known by now; its offsets load during this one
    const int64_t t_nx = (int64_t)__shfl_sync(FULL, g_next, 0);
    g_next = grab();
    int64_t nbeg = 0, nend = 0;
    if (t_nx < p.n_trials) {
      nbeg = __ldg(p.offsets + t_nx);
      nend = __ldg(p.offsets + t_nx + 1);
    }
    auto load_batch = [&](uint32_t e, int b, ulonglong2 (&v)[B]) {
#pragma unroll
      for (int u = 0; u < B; ++u) {
        const uint32_t eo = LPR == 1 ? e : __shfl_sync(FULL, e, (b * B + u) * RPW + lane / LPR);
        v[u] = make_ulonglong2(0ull, 0ull);
        if (eo != NONE) {
          if (K == 1) v[u].x = __ldg(p.table + eo);
          else v[u] = __ldg(reinterpret_cast<const ulonglong2*>(p.table) + (int64_t)eo * LPR + (lane % LPR));
        }
      }
    };
    auto use_batch = [&](ulonglong2 (&v)[B]) {
#pragma unroll
      for (int u = 0; u < B; ++u) {
        if (K == 1) {
          const bool c = (v[u].x & RW_CONT) != 0ull;
          push(c, v[u].x);
          if (c) v[u].x = 0ull;
          add_one(v[u].x);
        } else {
          const bool c = (v[u].y & RW_CONT) != 0ull;   // only ever in a row's last place
          push(c, v[u].y);
          if (c) v[u].y = (uint64_t)ns << 56;
          add_pair(v[u]);
        }
      }
    };
    ulonglong2 v[B];
    if (beg < end) load_batch(e_cur, 0, v);
    int rounds = 0;
    for (int64_t i0 = beg; i0 < end; i0 += 32) {
      const uint32_t e_nn = load_id(i0 + 64 + lane);
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        ulonglong2 vn[B];
        if (b + 1 < NB) load_batch(e_cur, b + 1, vn);
        else load_batch(e_nxt, 0, vn);
        use_batch(v);
#pragma unroll
        for (int u = 0; u < B; ++u) v[u] = vn[u];
      }
      e_cur = e_nxt;
      e_nxt = e_nn;
      if (++rounds == RW_SEG_ROUNDS) {
        __syncwarp();
        for (int i = lane; i < ns; i += 32) {
          const U128 S = drain(i);
          tot[i] = S.lo;
          tot[ns + i] = S.hi;
        }
        __syncwarp();
        rounds = 0;
      }
    }
    if (np) walk(np);
    const int64_t t_done = t;
    t = t_nx;
    beg = nbeg;
    end = nend;
    check_range();
    e_cur = load_id(beg + lane);                  // the next trial's first IDs load during the drain
    e_nxt = load_id(beg + 32 + lane);
    __syncwarp();
    for (int i = lane; i < ns; i += 32) {
      const U128 S = drain(i);
      tot[i] = 0ull;
      tot[ns + i] = 0ull;
      const LayerConst lc = p.layers[p.layer_of[i]];
      uint8_t reg;
      const double y = AccOps<U128>::finish(S, lc, reg);
      const int64_t at = (int64_t)i * p.n_trials + t_done;
      p.ylt[0][at] = y;
      if (p.regimes[0]) p.regimes[0][at] = reg;
    }
    __syncwarp();
  }
  if (bad_id) atomicOr(p.err, DERR_EVENT_RANGE);
  if (bad_off) atomicOr(p.err, DERR_OFFSETS);
}


// Rows end to end (K = 0), for long rows: the pairs of the rows of 32 occurrences are walked as one
// joined list, 32 pairs at a time.  A lane finds its pair's row from a bit mask of the rows that
// begin in the window (one warp OR) and the rank of the row among those with entries.
//
// PASSES: the pass reads every ID but keeps only the events in [e_lo, e_hi), whose rows stay in L2
// (compacted into a queue of 128 IDs per warp so that every round is full); the trial's exact
// sums go through `part` from one pass to the next.
//
// MULTI: requests with trial windows (RowsStream::windowed); otherwise one request over every trial.
template <int NC, bool MULTI, bool PASSES>
__global__ void __launch_bounds__(RW_WARPS * 32, RW_MIN_BLOCKS)
k_rows_join(RowsStream p) {
  constexpr uint32_t NONE = 0xffffffffu;
  extern __shared__ __align__(16) unsigned long long rw_smem[];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ns = p.ns;
  const uint32_t lt = (1u << lane) - 1u, le = lt | (1u << lane);
  const int words = (ns + 1) * NC + 2 * ns + 16 + (PASSES ? 64 : 0);
  unsigned long long* const acc0 = rw_smem + (int64_t)wid * words;
  unsigned long long* const tot = acc0 + (ns + 1) * NC;
  uint32_t* const rbase = reinterpret_cast<uint32_t*>(tot + 2 * ns);
  uint32_t* const queue = rbase + 32;             // [128], PASSES only
  unsigned long long* const col = acc0 + (lane & (NC - 1));
  const int rot = NC >= 16 ? lane : (NC == 8 ? lane >> 1 : lane >> 2);
  for (int i = lane; i < words; i += 32) acc0[i] = 0ull;
  __syncwarp();
  bool bad_id = false, bad_off = false;
  auto drain = [&](int i) -> U128 {
    U128 S{tot[i], tot[ns + i]};
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      unsigned long long* const a = acc0 + i * NC + ((c + rot) & (NC - 1));
      add_u64(S, *a);
      *a = 0ull;
    }
    return S;
  };
  auto grab = [&]() -> unsigned long long { return lane == 0 ? atomicAdd(p.queue, 1ull) : 0ull; };
  int64_t t = (int64_t)__shfl_sync(FULL, grab(), 0);
  unsigned long long g_next = grab();
  int64_t beg = 0, end = 0;
  if (t < p.n_trials) {
    beg = __ldg(p.offsets + t);
    end = __ldg(p.offsets + t + 1);
  }
  while (t < p.n_trials) {
    if (!(0 <= beg && beg <= end && end <= p.n_events)) { bad_off = true; beg = end = 0; }
    const int64_t t_nx = (int64_t)__shfl_sync(FULL, g_next, 0);
    g_next = grab();
    int64_t nbeg = 0, nend = 0;
    if (t_nx < p.n_trials) {
      nbeg = __ldg(p.offsets + t_nx);
      nend = __ldg(p.offsets + t_nx + 1);
    }
    uint32_t amask = 1u, sh_lo = 0u, sh_hi = 0u;
    if (MULTI) {
      amask = 0;
      for (int r = 0; r < p.n_req; ++r)
        if (t >= p.t0[r] && t < p.t1[r]) amask |= 1u << r;
      if (amask == 0u) end = beg;
      else {
        sh_lo = 8u * (uint32_t)(__ffs(amask) - 1);
        sh_hi = 8u * (uint32_t)(31 - __clz(amask));
      }
    }
    int64_t pos = beg;                            // next ID to read
    auto read_id = [&](int64_t i) -> uint32_t {
      if (i >= end) return NONE;
      const uint32_t e = (uint32_t)__ldcs(p.ids + i);
      if (e >= p.catalogue) { bad_id = true; return NONE; }
      return e;
    };
    int qh = 0, qn = 0;                           // queue head and length
    uint32_t ea = NONE, eb = NONE;                // IDs read ahead
    if (PASSES) {
      ea = read_id(pos + lane);
      eb = read_id(pos + 32 + lane);
    } else {
      ea = read_id(pos + lane);
    }
    auto next_round = [&]() -> uint32_t {         // event of this lane in the next round
      if constexpr (!PASSES) {
        const uint32_t e = ea;
        pos += 32;
        ea = read_id(pos + lane);
        return e;
      } else {
        while (qn < 32 && pos < end) {
          const uint32_t a = ea, b = eb;
          pos += 64;
          ea = read_id(pos + lane);
          eb = read_id(pos + 32 + lane);
          const bool ka = a - p.e_lo < p.e_n, kb = b - p.e_lo < p.e_n;   // NONE is in no range
          const uint32_t ma = __ballot_sync(FULL, ka), mb = __ballot_sync(FULL, kb);
          if (ka) queue[(qh + qn + __popc(ma & lt)) & 127] = a;
          qn += __popc(ma);
          if (kb) queue[(qh + qn + __popc(mb & lt)) & 127] = b;
          qn += __popc(mb);
        }
        __syncwarp();
        const int n = min(qn, 32);
        const uint32_t e = lane < n ? queue[(qh + lane) & 127] : NONE;
        qh += n;
        qn -= n;
        __syncwarp();
        return e;
      }
    };
    auto more = [&]() -> bool { return PASSES ? (qn > 0 || pos < end) : pos < end; };
    auto load_row = [&](uint32_t e) -> uint64_t { return e == NONE ? 0ull : __ldg(p.desc + e); };
    int rounds = 0;
    bool have = more();
    uint64_t ri_nxt = have ? load_row(next_round()) : 0ull;
    while (have) {
      const uint64_t ri = ri_nxt;
      have = more();
      if (have) ri_nxt = load_row(next_round());
      uint32_t cb, nch;
      if (MULTI) {
        const uint32_t incl_b = (uint32_t)(ri >> 32) * 0x01010101u;
        const uint32_t b0 = ((incl_b << 8) >> sh_lo) & 0xffu, b1 = (incl_b >> sh_hi) & 0xffu;
        cb = ((uint32_t)ri >> p.first_shift) + (b0 >> 1);
        nch = b1 > b0 ? ((b1 + 1u) >> 1) - (b0 >> 1) : 0u;
      } else {
        cb = (uint32_t)ri >> p.first_shift;
        nch = ((uint32_t)(ri >> 32) + 1u) >> 1;
      }
      uint32_t incl = nch;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += v;
      }
      const uint32_t total = __shfl_sync(FULL, incl, 31);
      const uint32_t excl = incl - nch;
      const uint32_t ne = __ballot_sync(FULL, nch != 0u);
      if (nch) rbase[__popc(ne & lt)] = cb - excl;
      __syncwarp();
      int started = -1;
      for (uint32_t w0 = 0; w0 < total; w0 += 32 * RW_U) {
        ulonglong2 v[RW_U];
#pragma unroll
        for (int u = 0; u < RW_U; ++u) {
          const uint32_t rel = excl - (w0 + 32u * u);
          const uint32_t m = __reduce_or_sync(FULL, (nch != 0u && rel < 32u) ? 1u << rel : 0u);
          const int own = started + __popc(m & le);
          started += __popc(m);
          const uint32_t x = w0 + 32u * u + (uint32_t)lane;
          v[u] = make_ulonglong2(0ull, 0ull);
          if (x < total) v[u] = __ldcg(reinterpret_cast<const ulonglong2*>(p.ovf) + (uint32_t)(rbase[own] + x));
        }
#pragma unroll
        for (int u = 0; u < RW_U; ++u) {
          if (u > 0 && w0 + 32u * u >= total) break;
          unsigned long long* const a = col + (uint32_t)(v[u].x >> 56) * NC;
          unsigned long long* const b = col + (uint32_t)(v[u].y >> 56) * NC;
          const unsigned long long qa = v[u].x & RW_Q, qb = v[u].y & RW_Q;
          add_columns<NC>(a, b, qa, qb, lane);
        }
      }
      __syncwarp();
      if (++rounds == 16) {
        for (int i = lane; i < ns; i += 32) {
          const U128 S = drain(i);
          tot[i] = S.lo;
          tot[ns + i] = S.hi;
        }
        __syncwarp();
        rounds = 0;
      }
    }
    for (int i = lane; i < ns; i += 32) {
      U128 S = drain(i);
      tot[i] = 0ull;
      tot[ns + i] = 0ull;
      const uint32_t r = MULTI ? (uint32_t)(i >= p.first[1]) + (uint32_t)(i >= p.first[2]) + (uint32_t)(i >= p.first[3]) : 0u;
      if (MULTI && !((amask >> r) & 1u)) continue;
      if (PASSES) {
        ulonglong2* const pt = p.part + t * ns + i;
        if (p.pass > 0) {
          const ulonglong2 o = __ldcs(pt);
          add_u128(S, o.x, o.y);
        }
        if (p.pass + 1 < p.n_pass) {
          __stcs(pt, make_ulonglong2(S.lo, S.hi));
          continue;
        }
      }
      const LayerConst lc = p.layers[p.layer_of[i]];
      uint8_t reg;
      const double y = AccOps<U128>::finish(S, lc, reg);
      const int64_t at = (int64_t)(i - p.first[r]) * (p.t1[r] - p.t0[r]) + (t - p.t0[r]);
      p.ylt[r][at] = y;
      if (p.regimes[r]) p.regimes[r][at] = reg;
    }
    __syncwarp();
    t = t_nx;
    beg = nbeg;
    end = nend;
  }
  if (bad_id) atomicOr(p.err, DERR_EVENT_RANGE);
  if (bad_off) atomicOr(p.err, DERR_OFFSETS);
}

// ------------------------------------------------------------------------------------------
// Host
// ------------------------------------------------------------------------------------------
bool rows_usable(const Portfolio& pf, const std::vector<int32_t>& sel) {
  if (!pf.d_ev_ptr || !pf.d_mem || sel.empty() || (int)sel.size() > RW_MAX_LAYERS) return false;
  std::vector<uint8_t> seen((size_t)pf.n_layers, 0);
  for (int32_t l : sel) {
    if (seen[(size_t)l] || !pf.layer_asc[(size_t)l]) return false;
    seen[(size_t)l] = 1;
  }
  return rows_sizes(pf, sel, 0).pairs < (int64_t)UINT32_MAX;
}

// Entries per event: an upper bound (every record of the layers) and a guess that counts an event
// once per layer and takes a third off for losses below the retentions.
static void row_entries(const Portfolio& pf, const std::vector<int32_t>& sel, int64_t* bound, double* likely) {
  *bound = 0;
  *likely = 0.0;
  const double C = (double)pf.catalogue;
  for (int32_t l : sel) {
    int64_t b = 0;
    for (int k = pf.layer_off[(size_t)l]; k < pf.layer_off[(size_t)l + 1]; ++k) {
      const size_t j = (size_t)pf.layer_elts[(size_t)k];
      b += pf.rec_off[j + 1] - pf.rec_off[j];
    }
    *bound += b;
    *likely += 0.65 * (1.0 - std::exp(-(double)b / C));
  }
}

// Entries kept in place per event: the power of two near the average row while the table stays
// within the part of L2 that serves random reads (about 64 MB here: a 128 MB table of the same rows
// ran at half the speed of a 64 MB one); longer rows lie end to end (K = 0).  Measured on 2.0-2.2e8
// occurrences over 2 M events, stream in ms:
//   0.19 entries per event, 30 layers: K = 1 1.35, K = 2 1.42, end to end 1.52
//   0.65, 8 layers: K = 2 1.29, K = 4 1.37, end to end 1.68
//   1.45, 16 layers: K = 4 1.31, K = 2 1.38, K = 1 1.72, end to end 1.70
//   6.2, 64 layers: K = 4 6.0, K = 8 6.9, end to end 4.3
int rows_k(const Portfolio& pf, const std::vector<int32_t>& sel) {
  int64_t bound;
  double likely;
  row_entries(pf, sel, &bound, &likely);
  const int K = likely < 0.3 ? 1 : likely < 1.0 ? 2 : likely < 2.2 ? 4 : 0;
  return 8 * (int64_t)K * pf.catalogue <= (80ll << 20) ? K : 0;
}

RowSizes rows_sizes(const Portfolio& pf, const std::vector<int32_t>& sel, int K) {
  RowSizes z;
  int64_t bound;
  row_entries(pf, sel, &bound, &z.likely_entries);
  const int64_t C = pf.catalogue;
  // K = 0: a pair per two entries and at most one half-empty pair per event.  Else the overflow of
  // rows longer than K: (n - K + 2) / 2 pairs, at most n / 2 (K >= 2) or 3 n / 4 (K = 1, n >= 2).
  z.pairs = K == 0 ? (bound + std::min(bound, C)) / 2 + 1 : K == 1 ? (3 * bound + 3) / 4 + 1 : bound / 2 + 1;
  z.first_shift = 2 * z.pairs < ((int64_t)1 << 32) ? 1 : 0;
  z.likely_bytes = 8 * C * std::max(K, 1) + (K == 0 ? (int64_t)(8.0 * (double)C * (z.likely_entries + 0.5)) : 0);
  return z;
}

// Columns: as many as leave 8 blocks per SM within about 190 KB of shared memory, because the rest
// is L1, where every row in flight holds a line (the 64-layer stream takes 4.3 ms with 8 columns and
// 60 KB of L1, 8.4 ms with 16 columns and 28 KB), but no more than a trial's entries fill: every
// column of every slot is read and cleared at the end of a trial.
// Passes: parts of the catalogue whose rows stay in L2 (118 MB of rows, 64 layers: 4.83 ms in one
// pass, 4.27 in two, 4.61 in three; 179 MB, 100 layers, 4 columns: 3.73 and 4.22; 283 MB, 150
// layers, 4 columns: 4.58 and 4.05).
RowSchedule rows_schedule(int ns, int K, int64_t table_bytes, double entries, int64_t n_trials, int64_t n_events) {
  RowSchedule r;
  const int extra = 16 * ns + (K > 0 ? 640 : 128);
  r.nc = 4;
  for (int nc : {8, 16, 32})
    if (8 * nc * (ns + 1) + extra <= 6144 && (nc < 32 || K > 0)) r.nc = nc;
  const double per_trial = entries * (double)n_events / (double)std::max<int64_t>(n_trials, 1);
  while (r.nc > 8 && (double)ns * r.nc > 4.0 * per_trial) r.nc /= 2;
  if (K == 0) {
    const int64_t one = r.nc >= 8 ? RW_PASS_BYTES + RW_PASS_BYTES / 3 : 3 * RW_PASS_BYTES;
    if (table_bytes > one) r.passes = 2;
  }
  return r;
}

static RowsBuild rows_build_params(const Portfolio& pf, const std::vector<int32_t>& sel) {
  RowsBuild p{};
  p.catalogue = pf.catalogue;
  p.ptr = pf.d_ev_ptr;
  p.elt = pf.d_ev_elt;
  p.loss = pf.d_ev_loss;
  p.elt_ret = pf.d_elt_ret;
  p.elt_lim = pf.d_elt_lim;
  p.mem = pf.d_mem;
  p.n_layers = pf.n_layers;
  p.layers = pf.d_layers;
  p.ns = (int32_t)sel.size();
  for (int i = 0; i < p.ns; ++i) {
    const int32_t l = sel[(size_t)i];
    p.slot_of[l] = (uint8_t)i;
    p.sel[l >> 6] |= 1ull << (l & 63);
  }
  return p;
}

template <bool ADJ>
static ara_status launch_build(const Portfolio& pf, const RowsBuild& p, cudaStream_t s) {
  ARA_TRY(cudaMemsetAsync(p.counters, 0, 2 * sizeof(uint32_t), s));
  const int smem = pf.n_layers * (int)sizeof(RowsLayer);
  const bool f32 = pf.d_rec_loss32 != nullptr;
  const auto fn = pf.n_layers <= 64 ? (f32 ? k_rows_build<float, 1, ADJ> : k_rows_build<double, 1, ADJ>)
                             : (f32 ? k_rows_build<float, 4, ADJ> : k_rows_build<double, 4, ADJ>);
  fn<<<(unsigned)((pf.catalogue + RW_BUILD_THREADS - 1) / RW_BUILD_THREADS), RW_BUILD_THREADS, smem, s>>>(p);
  ARA_TRY(cudaGetLastError());
  return ARA_OK;
}

ara_status launch_rows_build(Portfolio& pf, const std::vector<int32_t>& sel, const RowTable& rt, const int32_t* first,
                             cudaStream_t s) {
  RowsBuild p = rows_build_params(pf, sel);
  for (int i = 0; i < 5; ++i) p.first[i] = first[i];
  p.K = rt.K;
  p.table = rt.table;
  p.ovf = rt.ovf;
  p.ovf_pairs = rt.ovf_pairs;
  p.counters = rt.counters;
  p.desc = rt.desc;
  p.first_shift = rt.first_shift;
  return launch_build<false>(pf, p, s);
}

// Rows of the adjoint: cap entries at ent (in pairs), regimes zeroed by the caller, two counter words.
ara_status launch_adjoint_rows(const Portfolio& pf, const std::vector<int32_t>& sel, const AdjbSlots& q, uint32_t cap,
                               uint8_t* ent, uint64_t* desc, uint8_t* regime, uint32_t* counters, cudaStream_t s) {
  RowsBuild p = rows_build_params(pf, sel);
  p.ent = ent;
  p.desc = desc;
  p.regime = regime;
  p.q = q;
  p.ovf_pairs = cap / 2;
  p.counters = counters;
  return launch_build<true>(pf, p, s);
}

// Blocks per SM of a stream kernel with this much shared memory; ARA_ERANGE when it does not fit.
static ara_status rows_occupancy(const Portfolio& pf, const void* fn, int smem, int* per_sm) {
  if (smem > pf.max_smem_block) return ARA_ERANGE;
  const ara_status st = allow_shared(pf, fn);
  if (st != ARA_OK) return st;
  ARA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, fn, RW_WARPS * 32, smem));
  return *per_sm < 1 ? ARA_ERANGE : ARA_OK;
}

template <int NC, bool MULTI>
static ara_status launch_join(const Portfolio& pf, RowsStream p, RowSchedule& sched, cudaStream_t s) {
  const int passes = sched.passes;
  const auto fn = passes > 1 ? k_rows_join<NC, MULTI, true> : k_rows_join<NC, MULTI, false>;
  const int smem = RW_WARPS * ((p.ns + 1) * NC + 2 * p.ns + 16 + (passes > 1 ? 64 : 0)) * 8;
  int per_sm = 0;
  const ara_status st = rows_occupancy(pf, (const void*)fn, smem, &per_sm);
  if (st != ARA_OK) return st;
  sched.blocks = per_sm;
  const int64_t most = (p.n_trials + RW_WARPS - 1) / RW_WARPS;
  p.n_pass = passes;
  for (p.pass = 0; p.pass < passes; ++p.pass) {
    p.e_lo = (uint32_t)((uint64_t)p.catalogue * p.pass / passes);
    p.e_n = (uint32_t)((uint64_t)p.catalogue * (p.pass + 1) / passes) - p.e_lo;
    ARA_TRY(cudaMemsetAsync(p.queue, 0, sizeof(unsigned long long), s));
    fn<<<(unsigned)std::min<int64_t>(most, (int64_t)pf.n_sms * per_sm), RW_WARPS * 32, smem, s>>>(p);
    ARA_TRY(cudaGetLastError());
  }
  return ARA_OK;
}

static ara_status launch_rows_join(const Portfolio& pf, const RowsStream& p, RowSchedule& sched, cudaStream_t s) {
  const bool m = p.windowed;
  switch (sched.nc) {
    case 16: return m ? launch_join<16, true>(pf, p, sched, s) : launch_join<16, false>(pf, p, sched, s);
    case 8: return m ? launch_join<8, true>(pf, p, sched, s) : launch_join<8, false>(pf, p, sched, s);
    default: return m ? launch_join<4, true>(pf, p, sched, s) : launch_join<4, false>(pf, p, sched, s);
  }
}

template <int K, int NC>
static ara_status launch_stream(const Portfolio& pf, const RowsStream& p, RowSchedule& sched, cudaStream_t s) {
  const auto fn = k_rows_stream<K, NC>;
  const int smem = RW_WARPS * ((p.ns + 1) * NC + 2 * p.ns + RW_PEND + 16) * 8;
  int per_sm = 0;
  const ara_status st = rows_occupancy(pf, (const void*)fn, smem, &per_sm);
  if (st != ARA_OK) return st;
  sched.blocks = per_sm;
  const int64_t most = (p.n_trials + RW_WARPS - 1) / RW_WARPS;
  ARA_TRY(cudaMemsetAsync(p.queue, 0, sizeof(unsigned long long), s));
  fn<<<(unsigned)std::min<int64_t>(most, (int64_t)pf.n_sms * per_sm), RW_WARPS * 32, smem, s>>>(p);
  ARA_TRY(cudaGetLastError());
  return ARA_OK;
}

template <int K>
static ara_status launch_stream_nc(const Portfolio& pf, const RowsStream& p, RowSchedule& sched, cudaStream_t s) {
  switch (sched.nc) {
    case 32: return launch_stream<K, 32>(pf, p, sched, s);
    case 16: return launch_stream<K, 16>(pf, p, sched, s);
    case 8: return launch_stream<K, 8>(pf, p, sched, s);
    default: return launch_stream<K, 4>(pf, p, sched, s);
  }
}

// K > 0 holds the rows of one request over every trial; requests with windows always have their rows
// end to end, because the stream of rows in place writes every trial to d_ylt[0].
ara_status launch_rows_stream(Portfolio& pf, const RowsStream& p, int K, RowSchedule& sched, cudaStream_t s) {
  if (K > 0 && p.windowed) return ARA_EINVAL;
  switch (K) {
    case 1: return launch_stream_nc<1>(pf, p, sched, s);
    case 2: return launch_stream_nc<2>(pf, p, sched, s);
    case 4: return launch_stream_nc<4>(pf, p, sched, s);
    default: return launch_rows_join(pf, p, sched, s);
  }
}

}  // namespace ara
