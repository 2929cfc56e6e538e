"""The schedule of the few-subject alignment's strips, enumerated on the host
from the header that the kernel uses: the row between two strips crosses in a
ring (between two warps of a round) or a whole row (from the last warp of a
round to the first of the next), and CTA barriers between chunks of steps are
all that orders the warps."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Per length: the writer (lane 31 of a warp, column k - 31 at step k) and the
# reader (lane 0 of the warp below, column k at step k) of one row, chunk by
# chunk.  A column that is read must be the last one written to its slot, in an
# earlier chunk, and nothing may be written to the slot in the chunk that reads it.
PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "few_schedule.cuh"

struct Slot { int round, column, chunk; };

// the row between warps w and w + 1, or from the last warp to the next round's first
static bool row_ok(int L, int W, int w, int rounds) {
  const bool wraps = w + 1 == W;
  const int steps = few_steps(L), period = few_period(steps, W), slots = wraps ? L : kFewRing;
  std::vector<Slot> row(slots, Slot{-1, -1, -1});
  std::vector<int> read_in(slots, -1);
  const int total = rounds * period + W * kFewLag + steps;
  for (int g = 0; g < total; g += kFewStep) {
    int q = 0, k0 = 0;
    if (few_turn(g, wraps ? 0 : w + 1, period, q, k0) && k0 < steps && q < rounds)
      for (int k = k0; k < k0 + kFewStep && k < L; ++k) {
        if (wraps && q == 0) continue;  // the topmost strip has no row above
        const Slot &s = row[k % slots];
        read_in[k % slots] = g;
        if (s.round != (wraps ? q - 1 : q) || s.column != k || s.chunk >= g) return false;
      }
    if (few_turn(g, w, period, q, k0) && k0 < steps && q < rounds)
      for (int k = k0; k < k0 + kFewStep; ++k) {
        const int j = k - 31;
        if (j < 0 || j >= L) continue;
        if (read_in[j % slots] == g) return false;
        row[j % slots] = Slot{q, j, g};
      }
  }
  return true;
}

int main() {
  int bad = 0;
  for (int W = 1; W <= 16; ++W) {
    const int rounds = W == 16 ? 4 : 1;  // several rounds only with all sixteen warps
    for (int L = 1; L <= 8192; L += W == 16 || L < 1200 ? 1 : 61) {
      bool ok = W == 1 || row_ok(L, W, 0, rounds);
      if (W == 16) ok = ok && row_ok(L, W, 14, rounds) && row_ok(L, W, 15, rounds);
      if (!ok && ++bad <= 40) std::printf("L = %d, W = %d\n", L, W);
    }
  }
  return bad != 0;
}
"""


def test_no_row_is_read_before_or_after_its_time(tmp_path):
    src, exe = tmp_path / "schedule.cpp", tmp_path / "schedule"
    src.write_text(PROGRAM)
    inc = os.path.join(ROOT, "paper_1704_00878_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, "rows out of order at\n" + r.stdout
