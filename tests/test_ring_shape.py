"""The y,z ring's shape (ys::set_yz_grid, host code), over mesh sizes, grids and leads:

* S > D, so that a row item never waits for column items claimed after it (no deadlock);
* S never exceeds the slots allocated, nor the planes;
* where a slot is reused, S - D leaves a grid of items between a plane's columns and the
  rewrite of its slot;
* where there is a slot for every plane, the lead is the balanced one (up to the last plane).
"""
import json
import os
import subprocess

from paper_1505_05341_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "ys_internal.h"
namespace ys { int ring_lead_for(const Plan& p, int grid, int pct); void set_yz_grid(Plan& p, int grid, int lead_pct); }
int main() {
  const char* sep = "[";
  const int ns[] = {16, 32, 64, 96, 128, 192, 256, 512};
  for (int n : ns)
    for (int m = 1; m <= 2; ++m)
      for (int rows = 8; rows <= 32; rows *= 2)
        for (int cols = 1; cols <= 16; cols *= 4)
          for (int full = 152; full <= 304; full += 152) {
            ys::Plan p;
            p.n = n; p.m = m; p.nzc = n / 2; p.yz_rows = rows < n ? rows : n; p.yz_cols = cols;
            p.yz_w_row = 1.5 * 2.5 * rows; p.yz_w_col = 1.6 * 15 * cols; p.yz_grid_max = full;
            ys::set_yz_grid(p, full, ys::kRingLeadPctMax);
            const int cap = p.ring_slots_cap = p.ring_slots;
            for (int grid = full; grid >= full / 2; grid -= full / 4)
              for (int pct : {70, 100, 140, 200}) {
                ys::set_yz_grid(p, grid, pct);
                std::printf("%s[%d,%d,%d,%d,%d,%d,%d]", sep, n * m, cap, p.ring_slots, p.ring_lead,
                            ys::ring_lead_for(p, grid, pct), grid, n / p.yz_rows + (p.nzc + cols - 1) / cols);
                sep = ",";
              }
          }
  std::printf("]");
}
"""


def test_ring_shape(tmp_path):
    lib = build.build_library()
    src, exe = tmp_path / "ring.cu", tmp_path / "ring"
    src.write_text(PROGRAM)
    r = subprocess.run([build._nvcc(), *build.FLAGS, *build.ARCH, "-I", build.CSRC, "-I", os.path.join(build.HERE, "..", "include"),
                        "-o", str(exe), str(src), lib, "-Xlinker", "-rpath=" + os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rows = json.loads(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout)
    assert len(rows) > 1000
    for planes, cap, slots, lead, want, grid, items in rows:
        assert 1 <= lead < slots <= min(cap, planes), (planes, cap, slots, lead)
        if slots < planes:
            assert (slots - lead - 1) * items >= grid
        else:
            assert lead == min(want, planes - 1) or cap < planes or lead + 2 + -(-grid // items) <= planes
