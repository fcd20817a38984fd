"""The radial chunk rule of the tile kernels against a search over every chunk count (CPU)."""
import os
import shutil
import subprocess

import pytest

import paper_2609_21633_gb300 as tn

CSRC = os.path.join(os.path.dirname(os.path.abspath(tn.__file__)), "csrc")

MAIN = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
// the rule's divisions, counted through its cost function
static int64_t visits;
#define chunk_cost chunk_cost_plain
#include "radial_chunk_cost.inc"
#undef chunk_cost
namespace tn {
inline double chunk_cost(int64_t a, int b, int c, int d) { return ++visits, chunk_cost_plain(a, b, c, d); }
}
#include "radial_chunk_rule.inc"
int main() {
  const int64_t columns[] = {10, 40, 50, 160, 170, 640, 650, 2560, 10240};
  const int kmaxs[] = {1, 15, 32, 64, 128, 100000};
  for (int64_t col : columns)
    for (int resident = 1; resident <= 2; ++resident)
      for (int n = 0; n <= 1100; n += n < 140 ? 1 : 37)
        for (int kmax : kmaxs) {
          int best = 1;
          double cost = 1e30;
          for (int c = 1; c <= n; ++c) {
            const int kc = (n + c - 1) / c;
            if (kc > kmax) continue;
            const double t = tn::chunk_cost_plain(col, n, resident, kc);
            if (t < cost) cost = t, best = kc;
          }
          visits = 0;
          const int got = tn::radial_chunk(col, n, resident, kmax);
          if (got != best) return std::printf("columns %ld cells %d resident %d kmax %d: %d, not %d\n", (long)col, n, resident, kmax, got, best), 1;
          if (visits > 2 * std::sqrt((double)n) + 1) return std::printf("cells %d: %ld lengths visited\n", n, (long)visits), 2;
        }
  return 0;
}
"""


def test_same_chunk_as_the_full_search_in_few_steps(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("needs g++")
    text = open(os.path.join(CSRC, "radial_chunk.h")).read()
    head, rule = text.split("// Cell layers per radial chunk", 1)
    (tmp_path / "radial_chunk_cost.inc").write_text(head + "}\n")
    (tmp_path / "radial_chunk_rule.inc").write_text("namespace tn {\n//" + rule)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", str(tmp_path), str(tmp_path / "main.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], stdout=subprocess.PIPE, text=True)
    assert r.returncode == 0, r.stdout
