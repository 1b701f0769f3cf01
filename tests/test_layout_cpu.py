"""The shared-memory regions of a CTA's group levels nest (host build of csrc/layout.h).

Every group of a level moves on to the next level by itself, so the regions of
a group's sub-groups must lie inside the group's own region."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_02423_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "layout.h"
using namespace cfsim;
int main(int argc, char** argv) {
  const int nt = atoi(argv[1]), z = atoi(argv[2]);
  const ClassCfg c{nt, z, z / 2, z / 4, z / 8, (z / (nt / 32)) & ~15, kClassWarp, 0, 0, 0};
  int bad = 0;
  for (int w = 0; w < nt / 32; ++w) {
    const size_t lo = warp_region_at(w, c), hi = lo + c.z_wrp;
    const int e = w / (nt / 8 / 32);
    bad += lo % 16 != 0 || lo < (size_t)e * c.z_8th || hi > (size_t)(e + 1) * c.z_8th;
    if (w > 0) bad += lo < warp_region_at(w - 1, c) + c.z_wrp;
  }
  bad += 2 * c.z_8th > c.z_qtr || 2 * c.z_qtr > c.z_half || 2 * c.z_half > c.z_cta;
  printf("%d\n", bad);
  return 0;
}
"""


@pytest.mark.parametrize("nt", [512, 768, 1024])
def test_regions_nest(nt, tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe), str(nt), "225280"], check=True, capture_output=True, text=True).stdout == "0\n"
