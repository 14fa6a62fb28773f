"""The dX plan where the last vocabulary chunk is narrower than the others
(csrc/bgpo_plan.h): the estimate counts every chunk's own K blocks, and by the sum
over the chunks written out here no plan is slower than the usual one.
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

// K blocks of the longest split, chunk by chunk
static int64_t kblocks(const Geometry& g, int s) {
  int64_t n = 0;
  for (int64_t c = 0; c < g.n_vc; ++c)
    n += ceil_div(ceil_div(chunk_end(g, c) - chunk_begin(g, c), kBK), s);
  return n;
}

// the estimate with those K blocks (the other terms are the launches' and the partials')
static double cost(const Geometry& g, int64_t M, int pairs, const DxPlan& p) {
  const double waves =
      (double)ceil_div(ceil_div(M, kPairM) * dx_tiles_n(g.tiles_h, p.wide) * p.splits, pairs);
  const double block = p.wide == 1 ? 590 : 1030;
  return dx_cost(g, M, pairs, p.wide, p.splits) +
         waves * block * ((double)kblocks(g, p.splits) - (double)dx_kblocks(g, p.splits));
}

int main() {
  long bad = 0, wrong = 0, other = 0, narrow = 0;
  for (int64_t H : {304, 528, 1472, 1536, 3112, 4096})
    for (int64_t V : {700, 8193, 55165, 50001, 108141, 115266, 126464, 131046})
      for (int64_t rows : {125, 980, 1998, 5350})
        for (int64_t chunk : {0, 256, 4096, 8704, 13568, 15360, 16384}) {
          const Geometry g = make_geometry(1, 0, rows, H, V, chunk);
          const int64_t last = V - (g.n_vc - 1) * g.vc;
          narrow += g.n_vc > 1 && 8 * last < g.vc;
          for (int s = 1; s <= kMaxSplits; ++s) wrong += dx_kblocks(g, s) != kblocks(g, s);
          for (int64_t M : {rows / 6, rows / 2, rows}) {
            const DxPlan p = dx_plan(g, M, 76);
            const DxPlan u = {2, dx_splits(ceil_div(M, kPairM), dx_tiles_n(g.tiles_h), 76,
                                           g.kb_vc_min, dxp_row_block_cap(g))};
            if (p.wide == u.wide && p.splits == u.splits) continue;
            ++other;
            bad += cost(g, M, 76, p) > cost(g, M, 76, u);
          }
        }
  std::printf("%ld %ld %ld %ld\n", bad, wrong, other, narrow);
}
"""


def test_no_plan_is_slower_than_the_usual_one_by_the_chunks_own_k_blocks(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "chunks.cpp", tmp_path / "chunks"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    bad, wrong, other, narrow = map(
        int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert wrong == 0 and bad == 0
    assert other and narrow
