"""CPU check of the selection's launch plans (host arithmetic of csrc/ara_select_plan.h, compiled alone):
the allocation-free call's groups of rows cover the request and never need more than its fixed array."""
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
            if (y->bytes > limit || y->zero_bytes > y->bytes || y->n != n || y->n_t != t) ++bad;
            for (int i = 0; i < 12; ++i) bad += y->off[i] > y->off[i + 1] || y->off[i] % 16;
            if (y->off[12] + 8ull * y->n_layers * t > y->bytes) ++bad;
            if (!y->small && y->off[7] + 8ull * y->n_layers * t * y->cap > y->off[8]) ++bad;
          }
        }
  printf("%ld %ld\n", bad, uneven);
  return 0;
}
"""


def test_groups_of_the_allocation_free_call_fit_its_array(tmp_path):
    src, exe = tmp_path / "sweep.cpp", tmp_path / "sweep"
    src.write_text(SWEEP)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1606_04473_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    bad, uneven = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert bad == 0 and uneven > 1000
