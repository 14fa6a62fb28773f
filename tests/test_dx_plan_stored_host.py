"""The dX plan as the GEMM and the split reduction read it back (csrc/bgpo_plan.h,
dx_splits_stored, which both call, and dx_wide_stored): a plan that dx_plan makes
comes back as it is; a split count that does not fit the sample (too many for the
narrowest chunk's K blocks or for the split buffer) is one split for both, and
reported; a tile width that does not exist is one that does.
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
            bad += dx_splits_stored(g, M, p.splits, &fits) != p.splits || !fits;
            bad += dx_wide_stored(p.wide) != p.wide;
            for (int32_t wide : {-1, 0, 1, 2, 3, 0x5EED0000})
              bad += dx_wide_stored(wide) != (wide == 1 ? 1 : 2);
            for (int32_t s : {-0x7fffffff, -1, 0, 1, 2, 3, 5, 9, 15, 16, 17, 0x7fffffff}) {
              const bool ok = s >= 1 && s <= kMaxSplits && s <= g.kb_vc_min &&
                              s * ceil_div(M, kPairM) <= cap;
              bad += dx_splits_stored(g, M, s, &fits) != (ok ? s : 1) || fits != ok;
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
        assert sum("ERR_DX_SPLITS" in ln for ln in reads) == 1, (name, reads)
        assert all("dx_splits_stored(" in ln or "dx_wide_stored(" in ln for ln in reads), reads
