// few.cuh -- launch interface of the alignment to the center for few subjects
// (few.cu).
#pragma once
#include "sw_kernels.cuh"

struct FewJob {
  int center;                  // sorted index (or the view's)
  int sb, se;                  // subjects [sb, se), longest first
  uint16_t *codes;             // one slot of slot_codes entries per CTA
  size_t slot_codes;
  int2 *edge;                  // centers of more than kFewThreads / 32 strips: a row per CTA, else null
  int edge_cols;
  unsigned long long *counter; // zero
  const int32_t *perm;         // sorted index -> input index of the outputs
  uint16_t *ins;
  uint8_t *occ;
  int32_t *seg, *score;
  unsigned *err;
};

constexpr int kFewThreads = 512;  // at most; 32 per 128 center rows
constexpr int kFewRows = 4;       // center rows per lane

// 16-bit code words of a row of quads for a subject of L residues
__host__ __device__ __forceinline__ int few_row_slots(int L) { return (L + 31 + 15) & ~15; }
// code words of a CTA's slot
size_t few_slot_codes(int Lc, int maxlen);
// resident CTAs for n subjects (0: the center's profile does not fit)
int few_grid(int K, int Lc, int maxlen, int n);
// the center takes several rounds of strips (FewJob::edge is needed)
bool few_rounds(int Lc);
cudaError_t launch_align_few(const SeqSet &ss, const Scoring &sc, const FewJob &job, int Lc, int maxlen,
                             int grid, cudaStream_t st);
// modelled microseconds
double few_cost(int Lc, int n, double mean_len, int grid, int sms);
