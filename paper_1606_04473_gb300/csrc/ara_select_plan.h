// Launch plans of the PML / TVaR selection (ara_select.cu): its forms, block counts and scratch layout.
// Host arithmetic only, apart from the constants the kernels share.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace ara {

constexpr int SEL_THREADS = 512;
constexpr int SEL_SAMPLE = 1024;                 // sampled keys per row
constexpr int SEL_CLASSES = 2 * SEL_SAMPLE + 1;
constexpr int SEL_SMALL = 4096;                  // rows up to this length are sorted whole
// Rows of one request up to which they go as one cooperative launch.  Rows of 200,000 values, 3 targets / 6
// targets and the mean, us, cooperative and in clusters: 9 rows 43 / 60 and 47 / 62, 16 rows 56 / 72 and 83 / 106, 24
// rows 59 / 91 and 64 / 81, 32 rows 79 / 119 and 64 / 85, 64 rows 119 / 183 and 92 / 126.  (From about 24 rows
// clusters are the faster way since the keys take no FP64 instructions; the line decides the order in
// which TVaR and mean are added, and has stayed.)
constexpr int SEL_GRID_ROWS = 32;
constexpr int SEL_SLICES = 16;                   // slices of a row's sums that a block of a cluster can hold

struct SelState {
  uint64_t key;                // the selected key (known at once when its class is a tie)
  uint64_t lo, hi;             // the open interval it lies in otherwise (0 and ~0 at the ends: closed)
  int32_t tie;                 // 1: the class is a splitter's own
  int32_t list;                // the target whose list holds the interval (the first with that class)
  int64_t before;              // keys above the class
  int64_t in_class;            // keys in the class
};

// Sampled keys of a row, and room for the keys of one open interval between neighbouring samples: the
// interval that holds a given rank has 2 / sample of the keys on average and more than 16 / sample with
// probability 2e-6 (a list that would overflow is not used: its target is picked from the row itself).
// Sorting the sample costs every block 3.9 us for 256 keys and 6.7 for 1,024, and the intervals it leaves are
// picked from in about 4 us per 4,096 keys: 256 keys up to 2^19 values.
struct SelLists {
  int32_t sample;
  int64_t cap;                      // keys per list
};
inline SelLists roomy_lists(int64_t n) {
  const int32_t sample = n <= (1 << 19) ? 256 : SEL_SAMPLE;
  return SelLists{sample, std::min<int64_t>(n, 16 * (n / sample) + 4096)};
}
// The same chance of an overflow in up to eight times less room.
inline SelLists tight_lists(int64_t n) {
  return SelLists{SEL_SAMPLE, std::min<int64_t>(n, std::max<int64_t>(16 * (n / SEL_SAMPLE), SEL_SAMPLE))};
}

// A request's launch plan and scratch.  The form and the parts of a row that are summed one by one (on which
// the order of the TVaR and mean sums depends) follow from the request, the parts also where the form differs
// (beside).  How many rows share the lists at a time and how long the lists are follow from the memory, and
// change no result.
struct SelPlan {
  int64_t n = 0;
  SelLists lists{0, 0};
  int32_t n_layers = 0, n_t = 0, blocks = 1;
  int32_t slices = 1;               // parts of a row's sums, at least `blocks`
  int32_t per = 1;                  // rows per group; the groups run one after the other
  int32_t rounds = 1;               // 2: lists may well overflow, overfull intervals are split again before the pick
  bool cluster = false;             // one cluster of `blocks` blocks per row
  bool small = false;               // one block per row, sorted whole
  int n_sms = 1;
  // out and mean, err, then count, n_list, bar, count2, n_list2 (from err on cleared before the launch; err
  // only before the first group), state, list, psum, pmean, gt, eq
  size_t off[13];
  size_t zero_end = 0, bytes = 0;
  int32_t at_once() const { return std::max(1, (cluster ? 2 * n_sms : n_sms) / blocks); }   // rows that run at once
};
// per: 0 for all rows in one group.  beside: the caller's kernels share the device with other streams'
// (the server).  A row in a cluster whose list overflows is picked from the row itself, without a
// second round.
inline SelPlan sel_plan(int64_t n, int32_t n_layers, int32_t n_t, int n_sms, SelLists lists, bool beside = false,
                        int32_t per = 0) {
  SelPlan y;
  y.n = n;
  y.lists = lists;
  y.n_layers = n_layers;
  y.n_t = n_t;
  y.per = per > 0 ? std::min(per, n_layers) : n_layers;
  y.small = n <= SEL_SMALL;
  y.n_sms = std::max(1, n_sms);
  const int64_t slots = 2ll * y.n_sms;                      // blocks that run at once
  y.cluster = !y.small && n <= (4 << 20) && (beside || n_layers > SEL_GRID_ROWS);
  if (!y.small)
    y.slices = (int32_t)std::max<int64_t>(1, std::min<int64_t>((n + 2047) / 2048, std::max<int64_t>(1, n_sms / n_layers)));
  if (y.cluster) {                                          // all rows' clusters at once, if they can be
    y.blocks = 16;
    while (y.blocks > 1 && ((int64_t)n_layers * y.blocks > slots || n < 2048ll * y.blocks)) y.blocks /= 2;
    if (n_layers > SEL_GRID_ROWS) {
      y.slices = y.blocks;
    } else {       // the sums of the cooperative form, so that a served request's have the bits of a direct call's
      while (y.blocks > y.slices) y.blocks /= 2;
      if ((y.slices + y.blocks - 1) / y.blocks > SEL_SLICES) y.cluster = false;
    }
  }
  if (!y.cluster) y.blocks = y.slices;
  y.rounds = !y.small && !y.cluster && lists.cap < std::min<int64_t>(n, 16 * (n / lists.sample)) ? 2 : 1;
  const size_t L = (size_t)n_layers, lt = L * (size_t)n_t;
  const size_t G = (size_t)y.per, gt = G * (size_t)n_t, two = y.rounds > 1 ? gt : 0;   // of a group
  const size_t grid = y.small || y.cluster ? 0 : 1, listed = y.small ? 0 : 1;
  size_t b = 0;
  int i = 0;
  auto t = [&](size_t k, size_t align = 16) { b = (b + align - 1) / align * align; y.off[i++] = b; b += k; };
  t(8 * (lt + L));
  t(4, 8);                                                  // right behind the results: one copy takes both
  t(4 * grid * (n_t > 0 ? G : 0) * SEL_CLASSES);
  t(4 * grid * gt);
  t(4 * grid * G);
  t(4 * two * SEL_CLASSES);
  t(4 * two);
  y.zero_end = (b + 15) / 16 * 16;
  t(sizeof(SelState) * lt);
  t(8 * listed * gt * (size_t)lists.cap);
  t(8 * grid * gt * (size_t)y.blocks);
  t(8 * grid * G * (size_t)y.blocks);
  t(8 * lt);
  t(8 * lt);
  y.bytes = (b + 255) / 256 * 256;
  return y;
}

// A request's plan within `limit` bytes: roomy lists, else tight ones, else groups of rows (whole waves while
// they hold one), else shorter lists; the smallest plan where nothing fits.  1,000 rows of 200,000 values with
// 16 targets take 2.1 GB with roomy lists.
constexpr size_t SEL_SCRATCH = (size_t)4 << 30;
inline SelPlan sel_plan_within(int64_t n, int32_t n_layers, int32_t n_t, int n_sms, bool beside, size_t limit) {
  SelPlan y = sel_plan(n, n_layers, n_t, n_sms, roomy_lists(n), beside);
  if (y.bytes <= limit || y.small || n_t == 0) return y;
  SelLists lists = tight_lists(n);
  y = sel_plan(n, n_layers, n_t, n_sms, lists, beside);
  for (int32_t per = n_layers; y.bytes > limit && per > 1;) {
    per = (per + 1) / 2;
    if (per > y.at_once()) per -= per % y.at_once();
    y = sel_plan(n, n_layers, n_t, n_sms, lists, beside, per);
  }
  while (y.bytes > limit && lists.cap > SEL_SAMPLE) {
    lists.cap = std::max<int64_t>(lists.cap / 2, SEL_SAMPLE);
    y = sel_plan(n, n_layers, n_t, n_sms, lists, beside, 1);
  }
  return y;
}

// The allocation-free call within `limit` bytes: the request's own plan (roomy or tight lists) where it fits.
// Else its rows go as requests of their own, `per` at a time (plan `first`) and a last one of what is left
// (`last`), because fewer rows get more blocks each: in groups of one plan, 16 rows of 4.3 M values would run
// on 9 blocks at a time.  Where even one row's lists do not fit, shorter lists and a second round.  The last
// request can need more than the others although it has fewer rows (33 rows run as clusters, 32 as one
// cooperative launch with class counts), so both are checked.
struct SelGroups {
  int32_t per = 1;
  SelPlan first, last;
};
inline bool sel_groups(int64_t n, int32_t n_layers, int32_t n_t, int n_sms, size_t limit, SelGroups& g) {
  SelLists lists = roomy_lists(n);
  auto fits = [&](int32_t per) {
    g.per = per;
    g.first = sel_plan(n, per, n_t, n_sms, lists);
    g.last = n_layers % per ? sel_plan(n, n_layers % per, n_t, n_sms, lists) : g.first;
    return g.first.bytes <= limit && g.last.bytes <= limit;
  };
  if (fits(n_layers)) return true;
  lists = tight_lists(n);
  int32_t per = n_layers;
  while (!fits(per) && per > 1) per = (per + 1) / 2;
  while (!fits(per)) {
    if (lists.cap <= SEL_SAMPLE) return false;
    lists.cap = std::max<int64_t>(lists.cap / 2, SEL_SAMPLE);
  }
  return true;
}

}  // namespace ara
