"""The boundary rows of a center graph's launches, on the host: every launch that
may write them has an area of its own size, shared only with launches that it
cannot overlap."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# The full kernel writes a row after every pass but a pair's last, the bounded
# one after every pass: rows are written from two passes on, or from one on.
PROGRAM = r"""
#include <cstdio>
#include "center_rows.cuh"

int main() {
  int bad = 0;
  for (int npass = 1; npass <= 5; ++npass)
    for (int bounded = 0; bounded < 2; ++bounded) {
      const bool writes = (bounded ? npass : npass - 1) > 0, keeps = center_keeps_rows(npass, bounded);
      if (keeps != writes) std::printf("%d passes, bounded %d: keeps %d\n", npass, bounded, keeps), ++bad;
      for (int order = 0; order < 40; ++order) {
        const int lane = center_lane(order, keeps);
        if (lane < 0 || lane >= (writes ? kRowLanes : kCenterLanes)) std::printf("lane %d\n", lane), ++bad;
      }
    }
  return bad != 0;
}
"""


def test_launches_that_write_rows_have_an_area(tmp_path):
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_1704_00878_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
