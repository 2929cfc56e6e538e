// few_schedule.cuh -- when each warp of the few-subject alignment (few.cu)
// sweeps which strip of center rows.  Plain C++ beside the qualifiers, so the
// host can enumerate the schedule.
#pragma once

#ifdef __CUDACC__
#define FEW_FN __host__ __device__ __forceinline__
#else
#define FEW_FN inline
#endif

constexpr int kFewStep = 16;  // steps between CTA barriers (a chunk)
constexpr int kFewLag = 48;   // steps a strip runs behind the one above: 31 + 16, rounded up
constexpr int kFewRing = 64;  // columns of the row between two strips

static_assert(kFewLag % kFewStep == 0 && kFewLag >= 31 + kFewStep, "a column must be complete a barrier before it is read");
static_assert(kFewRing >= kFewLag - 31 + 2 * kFewStep, "ring");

// Steps of a strip against a subject of L residues: 31 to fill the lanes, whole
// chunks.
FEW_FN int few_steps(int L) { return (L + 31 + kFewStep - 1) / kFewStep * kFewStep; }

// Steps from a warp's strip to its next one, W strips further down.  The row
// above that one comes from the last warp of this round, W * kFewLag steps
// behind at most.  And the warp's own ring starts again at slot 0 when its next
// strip has column 0 (step 31, in the second chunk), while the warp below
// reads the last column of this round at step L - 1 + kFewLag: with no more than
// `steps` between two strips both fall into one chunk where L = 1 (mod 64), the
// slots are the same and no barrier lies between.  One more chunk puts the
// reader a barrier ahead at every length.
FEW_FN int few_period(int steps, int W) {
  const int wrap = steps + kFewStep, down = W * kFewLag;
  return wrap > down ? wrap : down;
}

// The strip (round q of warp w's, step k0 of it) that warp w sweeps in the chunk
// at step g of the CTA; false before its first one.
FEW_FN bool few_turn(int g, int w, int period, int &q, int &k0) {
  const int rel = g - w * kFewLag;
  if (rel < 0) return false;
  q = rel / period;
  k0 = rel - q * period;
  return true;
}
