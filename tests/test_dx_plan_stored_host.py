"""The dX plan as the GEMM and the split reduction read it back (csrc/bgpo_plan.h,
dx_plan_stored, which both call): a plan that dx_plan makes comes back as it is;
any other pair of words that does not fit the sample (too many splits for the
narrowest chunk's K blocks or for the split buffer, a tile width that does not
exist) is an unsplit plan for both, and reported.
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
  long bad = 0, good = 0, refused = 0, kblocks = 0;
  for (int64_t H : {64, 136, 1024, 4096})
    for (int64_t V : {1, 65, 975, 8192})
      for (int64_t rows : {1, 33, 2048})
        for (int64_t chunk : {0, 256, 4096}) {
          const Geometry g = make_geometry(1, 0, rows, H, V, chunk);
          const int64_t cap = dxp_row_block_cap(g);
          for (int64_t M : {int64_t(1), rows}) {
            const DxPlan p = dx_plan(g, M, 76);
            bool fits = false;
            const DxPlan q = dx_plan_stored(g, M, p.wide, p.splits, &fits);
            bad += !fits || q.wide != p.wide || q.splits != p.splits;
            for (int32_t wide : {-1, 0, 1, 2, 3, 0x5EED0000})
              for (int32_t s : {-0x7fffffff, -1, 0, 1, 2, 3, 5, 9, 15, 16, 17, 0x7fffffff}) {
                const DxPlan r = dx_plan_stored(g, M, wide, s, &fits);
                const bool ok = (wide == 1 || wide == 2) && s >= 1 && s <= kMaxSplits &&
                                s <= g.kb_vc_min && s * ceil_div(M, kPairM) <= cap;
                bad += ok != fits;
                bad += ok ? (r.wide != wide || r.splits != s) : r.splits != 1;
                bad += r.wide != 1 && r.wide != 2;
                good += ok;
                refused += !ok;
                kblocks += s >= 1 && s <= kMaxSplits && s > g.kb_vc_min;
              }
          }
        }
  std::printf("%ld %ld %ld %ld\n", bad, good, refused, kblocks);
}
"""


def test_the_gemm_and_the_reduction_read_one_plan(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "stored.cpp", tmp_path / "stored"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", f"-I{CSRC}", str(src), "-o", str(exe)], check=True)
    bad, good, refused, kblocks = map(
        int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert bad == 0
    assert good and refused and kblocks
    # neither kernel reads the words any other way
    for name in ("k_gemm.cu", "k_small.cu"):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        reads = [ln for ln in text.splitlines() if "err[ERR_DX_" in ln and "] = " not in ln]
        assert len(reads) == 1 and "dx_plan_stored" in text, (name, reads)
