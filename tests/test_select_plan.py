"""CPU checks of the selection's launch plans (host arithmetic of csrc/ara_select_plan.h, compiled alone):
the allocation-free call's groups of rows cover the request and never need more than its fixed array;
with less memory the other calls take fewer rows at a time and shorter lists in the same form."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SWEEP = r"""
#include <stdio.h>
#include "ara_select_plan.h"
using namespace ara;
int main() {
  const size_t limit = 4u << 20;
  long bad = 0, uneven = 0;
  const int64_t ns[] = {1, 64, 4096, 4097, 5000, 9999, 19052, 30011, 57935, 100003, 200000, 524288, 524289, 1000000,
                        4194304, 4194305, 10000000, 300000000};
  for (int sms : {1, 7, 148, 152})
    for (int64_t n : ns)
      for (int L = 1; L <= 300; ++L)
        for (int t = 0; t <= 16; ++t) {
          if (8192u * L * t > limit) continue;        // refused before any plan
          SelGroups g;
          if (!sel_groups(n, L, t, sms, limit, g)) { ++bad; continue; }
          const int left = L % g.per;
          uneven += left != 0;
          if (g.per < 1 || g.per > L || g.first.n_layers != g.per || g.last.n_layers != (left ? left : g.per)) ++bad;
          for (const SelPlan* y : {&g.first, &g.last}) {
            if (y->bytes > limit || y->zero_end > y->off[7] || y->n != n || y->n_t != t) ++bad;
            for (int i = 0; i < 12; ++i) bad += y->off[i] > y->off[i + 1] || y->off[i] % 8;
            if (y->off[12] + 8ull * y->n_layers * t > y->bytes) ++bad;
            if (!y->small && y->off[8] + 8ull * y->n_layers * t * y->lists.cap > y->off[9]) ++bad;
          }
        }
  printf("%ld %ld\n", bad, uneven);
  return 0;
}
"""


WITHIN = r"""
#include <stdio.h>
#include "ara_select_plan.h"
using namespace ara;
int main() {
  long bad = 0, grouped = 0, shorter = 0;
  const int64_t ns[] = {1, 4096, 4097, 30011, 200000, 1000000, 4194305, 10000000};
  const size_t limits[] = {0, 100000, 1000000, 30000000, SEL_SCRATCH};
  for (int64_t n : ns)
    for (int L : {1, 2, 6, 32, 33, 64, 100, 152, 304, 1000, 100000})
      for (int t = 0; t <= 16; ++t)
        for (int beside = 0; beside < 2; ++beside) {
          const SelPlan all = sel_plan(n, L, t, 152, roomy_lists(n), beside);
          size_t before = 0;
          for (size_t limit : limits) {
            const SelPlan y = sel_plan_within(n, L, t, 152, beside, limit);
            // the results' order of addition follows from the request alone
            bad += y.blocks != all.blocks || y.cluster != all.cluster || y.small != all.small;
            bad += y.bytes > all.bytes + 8 * 16 * SEL_CLASSES + 4096 || y.bytes < before || y.per < 1 || y.per > L;
            if (limit >= all.bytes) bad += y.per != L || y.lists.cap != all.lists.cap || y.rounds != all.rounds;
            if (y.bytes <= limit && y.per > y.at_once() && y.per < L) bad += y.per % y.at_once() != 0;
            // never much more than 8 KiB for each row and target and the results
            if (limit == 0) bad += y.bytes > 17000ull * (t + 1) + 100ull * L * (t + 1) + 8ull * 152 * (t + 1) + 4096;
            for (int i = 0; i < 12; ++i) bad += y.off[i] > y.off[i + 1] || y.off[i] % 8;
            if (!y.small && y.off[8] + 8ull * y.per * t * y.lists.cap > y.off[9]) ++bad;
            grouped += y.per < L;
            shorter += y.lists.cap < all.lists.cap;
            before = y.bytes;
          }
        }
  printf("%ld %ld %ld\n", bad, grouped, shorter);
  return 0;
}
"""


def sweep(tmp_path, text):
    src, exe = tmp_path / "sweep.cpp", tmp_path / "sweep"
    src.write_text(text)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1606_04473_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    return list(map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()))


def test_plans_within_less_memory_keep_the_form(tmp_path):
    bad, grouped, shorter = sweep(tmp_path, WITHIN)
    assert bad == 0 and grouped > 1000 and shorter > 1000


def test_groups_of_the_allocation_free_call_fit_its_array(tmp_path):
    bad, uneven = sweep(tmp_path, SWEEP)
    assert bad == 0 and uneven > 1000
