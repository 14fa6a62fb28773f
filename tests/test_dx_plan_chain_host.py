"""How long a chain of additions the dX plan gives an fp32 accumulator
(csrc/bgpo_plan.h): no longer than the usual plan's, or at most 16 K blocks. The
rounding error of dX's sums grows with the chain.
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
// the longest K loop of any split in any chunk, in K blocks, as the GEMM cuts it
static int64_t chain(const Geometry& g, int splits) {
  int64_t most = 0;
  for (int64_t c = 0; c < g.n_vc; ++c) {
    const int64_t kb = ceil_div(chunk_end(g, c) - chunk_begin(g, c), kBK);
    for (int64_t s = 0; s < splits; ++s) {
      const int64_t n = (s + 1) * kb / splits - s * kb / splits;
      if (n > most) most = n;
    }
  }
  return most;
}
int main() {
  long bad = 0, fewer = 0, other = 0;
  for (int64_t H : {64, 304, 1024, 1536, 2712, 4096})
    for (int64_t V : {65, 500, 1000, 1100, 8192, 50001, 126464, 152064})
      for (int64_t rows : {33, 256, 980, 2048, 8192, 32768})
        for (int64_t chunk : {0, 256, 1024, 1280, 13568}) {
          const Geometry g = make_geometry(1, 0, rows, H, V, chunk);
          for (int64_t M : {rows / 26, rows / 8, rows / 2, rows}) {
            if (M <= 0) continue;
            const DxPlan p = dx_plan(g, M, 76);
            const int usual = dx_splits(ceil_div(M, kPairM), dx_tiles_n(g.tiles_h), 76,
                                        g.kb_vc_min, dxp_row_block_cap(g));
            bad += chain(g, p.splits) > chain(g, usual) && chain(g, p.splits) > 16;
            fewer += p.splits < usual;
            other += p.wide != 2 || p.splits != usual;
          }
        }
  std::printf("%ld %ld %ld\n", bad, fewer, other);
}
"""


def test_accumulator_chains_are_no_longer_than_the_usual_plans(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "chain.cpp", tmp_path / "chain"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    bad, fewer, other = map(
        int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert bad == 0
    assert fewer and other > fewer
