"""Host-side invariants of the dX GEMM's plan (csrc/bgpo_plan.h, dx_plan): the tile
width and split count always fit the split buffer and the K blocks, the usual
plan stands unless the other is estimated to take at least 5% less, and a large
head without chunks keeps it.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2510_11683_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "bgpo_plan.h"
using namespace bgpo;
int main() {
  long bad = 0, n = 0, kept = 0, one = 0, unsplit = 0;
  for (int64_t H : {64, 136, 256, 264, 1024, 2712, 4096, 16384})
    for (int64_t V : {1, 64, 65, 975, 8192, 50001, 126464})
      for (int64_t rows : {1, 33, 256, 2048, 8192})
        for (int64_t chunk : {0, 256, 8192})
          for (int pairs : {1, 7, 74, 76}) {
            const Geometry g = make_geometry(1, 0, rows, H, V, chunk);
            const int64_t cap = dxp_row_block_cap(g);
            for (int64_t M : {int64_t(0), int64_t(1), rows / 2, rows}) {
              const DxPlan p = dx_plan(g, M, pairs);
              const int64_t mb = ceil_div(M, kPairM);
              ++n;
              bad += !(p.wide == 1 || p.wide == 2) || p.splits < 1 || p.splits > kMaxSplits;
              if (M <= 0) { bad += p.splits != 1; continue; }
              bad += p.splits * mb > cap || p.splits > g.kb_vc_min;
              const int usual = dx_splits(mb, dx_tiles_n(g.tiles_h), pairs, g.kb_vc_min, cap);
              if (p.wide == 2 && p.splits == usual) { ++kept; continue; }
              bad += dx_cost(g, M, pairs, p.wide, p.splits) >
                     0.951f * dx_cost(g, M, pairs, 2, usual);
              one += p.wide == 1;
              unsplit += p.splits == 1;
            }
          }
  // a large head at every sample size of a batch
  long big = 0;
  const int64_t heads[][4] = {{8, 256, 4096, 126464}};
  for (const auto& h : heads)
    for (int64_t M = 256; M <= h[0] * h[1]; M += 256) {
      const Geometry g = make_geometry(h[0], 0, h[1], h[2], h[3]);
      const DxPlan p = dx_plan(g, M, 76);
      big += p.wide != 2 || p.splits != dx_splits(ceil_div(M, kPairM), dx_tiles_n(g.tiles_h), 76,
                                                  g.kb_vc_min, dxp_row_block_cap(g));
    }
  std::printf("%ld %ld %ld %ld %ld %ld\n", bad, n, kept, one, unsplit, big);
}
"""


def test_dx_plan_fits_and_improves(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    bad, n, kept, one, unsplit, big = map(
        int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert bad == 0 and n > 10000
    assert kept and one and unsplit     # every kind of plan occurs
    assert big == 0
