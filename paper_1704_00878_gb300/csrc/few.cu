// few.cu -- alignment to the center for few subjects: fill, traceback codes
// and the traceback itself in one launch, one CTA per subject.
//
// The codes kernels give each subject (or pair of them) one group of at most
// 32 lanes and 16 center rows per lane: best when thousands of subjects fill
// the chip, but a few hundred leave most schedulers idle and a subject's
// passes run one after another.  Here a CTA spreads one subject's rows over
// up to 16 warps, 4 rows per lane, so that what bounds a subject is its
// wavefront (columns + ramps) and not its cells:
//   - warp w takes the strip of 128 center rows w, w + W, ...; its lanes sweep
//     the columns as an anti-diagonal wavefront (bottom rows move down a lane
//     by shuffle);
//   - the warps run in lockstep chunks of 16 steps, each 48 steps behind the
//     one above it, so the row between two strips crosses in a 64-column ring
//     in shared memory, and one CTA barrier per chunk is all the
//     synchronisation; between rounds of W strips the row sits in global
//     memory;
//   - codes: 16 bits per column for a lane's 4 rows, column j of quad q in slot
//     j + (q mod 32) -- the lane's step -- so a lane writes 32 bytes per chunk;
//     code 0 marks H = 0, so the traceback needs the codes alone;
//   - the traceback follows in the same CTA: a warp copies 32 quads x 128
//     columns around the path into shared memory and walks them there.
// int32 cells (any center).  Measured on one GB300, alignment stage with the
// traceback: 240 proteins of 900-5,000 residues 5.4 ms (one warp per subject,
// 16 rows per lane: 48.6); 200 of 200-400 residues 93 us (514); 24 of 30-120
// 31 us (120).
#include <algorithm>

#include "dp_pass.cuh"
#include "few.cuh"
#include "few_schedule.cuh"

namespace {

constexpr int kR = kFewRows;               // center rows per lane
constexpr int kStrip = 32 * kR;            // rows of a warp's strip
constexpr int kStep = kFewStep, kLag = kFewLag, kRing = kFewRing;
constexpr int kTileCols = 128, kTileSlots = kTileCols + 8;  // traceback window: columns, 16-byte aligned slots

// a lane's state while its warp sweeps a strip
struct FewLane {
  int H[kR], E[kR], rb[kR], rj[kR], be[kR];
  int hbot, fbot, htop;
};

__global__ void __launch_bounds__(kFewThreads, 1) k_align_few(SeqSet ss, Scoring sc, FewJob job) {
  extern __shared__ __align__(16) int8_t smem[];
  __shared__ int8_t sM[MSA_MAX_ALPHABET * MSA_MAX_ALPHABET];
  __shared__ __align__(16) uint16_t s_tile[32 * kTileSlots];
  __shared__ int2 s_ring[kFewThreads / 32][kRing];
  __shared__ unsigned long long s_best;
  __shared__ int s_item;
  const int K = sc.K, padc = K, o = sc.o, e = sc.e;
  const int NT = (int)blockDim.x, W = NT >> 5, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int Lc = ss.len[job.center];
  const uint8_t *rc = ss.res + ss.pstart[job.center];
  const int nstrip = (Lc + kStrip - 1) / kStrip, rows = nstrip * kStrip;
  int8_t *prof = smem;                                     // (K + 1) x rows: s + o, padding 0
  uint8_t *sres = reinterpret_cast<uint8_t *>(smem) + (size_t)(K + 1) * rows;
  for (int i = tid; i < K * K; i += NT) sM[i] = sc.M[i];
  __syncthreads();
  for (int idx = tid; idx < (K + 1) * (rows / 4); idx += NT) {
    const int r = idx / (rows / 4), i = 4 * (idx - r * (rows / 4));
    uint32_t v = 0;
    if (r < K)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i + u < Lc) v |= (uint32_t)(uint8_t)(sM[rc[i + u] * K + r] + o) << (8 * u);
    reinterpret_cast<uint32_t *>(prof)[idx] = v;
  }
  uint16_t *codes = job.codes + (size_t)blockIdx.x * job.slot_codes;
  int2 *edge = job.edge ? job.edge + (size_t)blockIdx.x * job.edge_cols : nullptr;
  for (;;) {
    __syncthreads();  // the last subject's shared state is done with
    if (tid == 0) {
      s_item = (int)atomicAdd(job.counter, 1ull);
      s_best = 0ull;
    }
    __syncthreads();
    const int item = s_item;
    if (item >= job.se - job.sb) break;
    const int kx = job.se - 1 - item;  // longest first
    const int L = ss.len[kx];
    const uint8_t *rs = ss.res + ss.pstart[kx];
    for (int i = tid; i < L; i += NT) sres[i] = rs[i];
    const int row_slots = few_row_slots(L);
    const int steps = few_steps(L), period = few_period(steps, W);
    const int rounds = (nstrip + W - 1) / W;
    const int total = (rounds - 1) * period + ((nstrip - 1) % W) * kLag + steps;
    __syncthreads();
    FewLane s;
    unsigned long long key = 0ull;
    for (int g = 0; g < total; g += kStep) {
      int q = 0, k0 = 0;
      const bool on = few_turn(g, w, period, q, k0);
      const int strip = q * W + w;
      if (on && k0 < steps && strip < nstrip) {
        if (k0 == 0) {
#pragma unroll
          for (int r = 0; r < kR; ++r) { s.H[r] = 0; s.E[r] = 0; s.rb[r] = 0; s.rj[r] = 0; s.be[r] = 0; }
          s.hbot = s.fbot = s.htop = 0;
        }
        const int8_t *pb = prof + strip * kStrip + lane * kR;
        const bool last = strip + 1 == nstrip;
        uint32_t *dst = reinterpret_cast<uint32_t *>(codes + (size_t)(strip * 32 + lane) * row_slots + k0);
        const bool mine = strip * kStrip + lane * kR < Lc;
        // four steps at a time: their profile words and the row above first,
        // then the cells, then the row below and the codes (a longer unrolled
        // body runs out of the instruction cache; loads behind the ring's
        // stores would wait for them)
#pragma unroll 1
        for (int u0 = 0; u0 < kStep; u0 += 4) {
          uint32_t pws[4], cw[2];
          int2 above[4], below[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int k = k0 + u0 + u, j = k - lane;
            const int res = (unsigned)j < (unsigned)L ? sres[j] : padc;
            pws[u] = *reinterpret_cast<const uint32_t *>(pb + res * rows);
            above[u] = make_int2(0, 0);
            if (lane == 0 && strip > 0 && k < L) above[u] = w > 0 ? s_ring[w - 1][k & (kRing - 1)] : __ldcg(edge + k);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = k0 + u0 + u - lane;
            int hin = __shfl_up_sync(MSA_FULL_MASK, s.hbot, 1), fin = __shfl_up_sync(MSA_FULL_MASK, s.fbot, 1);
            if (lane == 0) {
              hin = above[u].x;
              fin = above[u].y;
            }
            const uint32_t pw = pws[u];
            // E* = E + o and F* = F + o as in the codes kernels, but F* of the next
            // row from q = max(P, E*) - o (or 0) alone: H = max(q, F* - o), and
            // F* - e >= F* - o, so the rows' serial chain is one instruction each
            int hdiag = s.htop, hup = hin, f = __viaddmax_s32(fin, -e, hin);
            s.htop = hin;
            const int jm = max(j, 0);  // (before its first column a lane's cells are all 0)
            uint32_t code = 0;
            // flags as differences of ordered values, clamped to 1, and put
            // together by multiply-adds: comparisons and selections take twice
            // the integer pipe's time of an addition or a two-operand minimum
            Unroll<kR>::run([&](auto ic) {
              constexpr int r = decltype(ic)::value;
              const int p = hdiag + Cell<false>::template score<r & 3>(pw, 0u);
              const int pe = max(p, s.E[r]);
              const int q = __viaddmax_s32_relu(pe, -o, 0);
              const int hv = __viaddmax_s32(f, -o, q);
              const int m = max(pe, f);
              // source: 1 diagonal, 2 F, 3 E (ties in that order), 0 where H = 0
              const int a = min(m - p, 1), x = min(m - f, a), z = min(hv, 1);
              const uint32_t src = mad_lo((uint32_t)(a + x), (uint32_t)z, (uint32_t)z);
              const uint32_t bf = (uint32_t)min(f - hup, 1);  // F extended
              code = mad_lo(mad_lo(bf, 8u, mad_lo((uint32_t)s.be[r], 4u, src)), 1u << (4 * r), code);
              if constexpr (r == kR - 1) s.fbot = f;  // (the lane below extends it itself)
              f = __viaddmax_s32(f, -e, q);  // F* of the row below
              s.E[r] = __viaddmax_s32(s.E[r], -e, hv);
              s.be[r] = min(s.E[r] - hv, 1);  // E extended, in the next column
              const int rbn = max(s.rb[r], hv);
              s.rj[r] = max(s.rj[r], (int)mad_lo((uint32_t)min(rbn - s.rb[r], 1), (uint32_t)jm, 0u));
              s.rb[r] = rbn;
              hdiag = s.H[r];
              s.H[r] = hv;
              hup = hv;
            });
            s.hbot = hup;
            if (u & 1) cw[u >> 1] |= code << 16;
            else cw[u >> 1] = code;
            below[u] = make_int2(s.hbot, s.fbot);
          }
          if (lane == 31 && !last) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int j = k0 + u0 + u - 31;
              if ((unsigned)j >= (unsigned)L) continue;
              if (w + 1 < W) s_ring[w][j & (kRing - 1)] = below[u];
              else __stcg(edge + j, below[u]);
            }
          }
          if (mine) *reinterpret_cast<uint2 *>(dst + u0 / 2) = make_uint2(cw[0], cw[1]);
        }
        if (k0 + kStep >= steps) {
#pragma unroll
          for (int r = 0; r < kR; ++r) {
            const unsigned long long c = best_key(s.rb[r], strip * kStrip + lane * kR + r + 1, s.rj[r] + 1);
            key = c > key ? c : key;
          }
        }
      }
      __syncthreads();
    }
    if (key) atomicMax(&s_best, key);
    __syncthreads();
    if (w != 0) continue;

    // ---- traceback (one warp, every lane the same walk)
    const unsigned long long bk = s_best;
    const int bv = best_key_score(bk), i2 = best_key_row(bk), j2 = best_key_col(bk);
    const int orig = job.perm[kx];
    uint16_t *in = job.ins + (size_t)orig * (Lc + 1);
    uint8_t *oc = job.occ + (size_t)orig * (Lc + 1);
    int i = i2, j = j2;
    bool ok = bv <= 0;
    if (bv > 0 && (i2 > Lc || j2 > L)) {  // a best cell outside the matrix
      if (lane == 0) atomicOr(job.err, MSA_DERR_TRACE);
      continue;
    }
    // the lanes look ahead along the path's direction (diagonal in state H, up
    // in F, left in E), so a run of equal steps is one turn of the loop
    int state = 0, left = 2 * (i2 + j2) + 64;  // state: 0 = H, 1 = F, 2 = E
    int pending = 0;                           // E steps at center row i
    while (!ok && left > 0) {
      // the window: quads q0 .. q0 + 31 (rows up to i), columns c0 .. j (1-based)
      const int q1 = (i - 1) >> 2, q0 = max(0, q1 - 31), c0 = max(1, j - kTileCols + 1);
      __syncwarp();
      {
        const int q = q0 + lane;
        if (q <= q1) {
          const int s0 = (c0 - 1 + (q & 31)) & ~7;
          const uint4 *src = reinterpret_cast<const uint4 *>(codes + (size_t)q * row_slots + s0);
          uint4 *dst = reinterpret_cast<uint4 *>(s_tile + lane * kTileSlots);
          const int chunks = ((j - 1 + (q & 31)) - s0) / 8 + 1;
#pragma unroll
          for (int c = 0; c < kTileSlots / 8; ++c)
            if (c < chunks) dst[c] = __ldcg(src + c);
        }
      }
      __syncwarp();
      const int row_min = 4 * q0;  // rows > row_min and columns >= c0 are in the window
      while (i > row_min && j >= c0 && left > 0) {
        --left;
        const int ri = state == 2 ? i : i - lane, cj = state == 1 ? j : j - lane;
        const bool in_win = ri > row_min && cj >= c0;
        uint32_t code = 0;
        if (in_win) {
          const int q = (ri - 1) >> 2, sk = q & 31;
          code = s_tile[(q - q0) * kTileSlots + (cj - 1 + sk) - ((c0 - 1 + sk) & ~7)] >> (4 * ((ri - 1) & 3));
        }
        const bool go = in_win && (state == 0 ? (code & 3u) == 1u : ((code >> (state == 1 ? 3 : 2)) & 1u) != 0);
        const unsigned stops = ~__ballot_sync(MSA_FULL_MASK, go);
        const int run = stops ? __ffs(stops) - 1 : 32;  // lanes that go on
        // the lane that does not: out of the window, or the run's last cell
        const unsigned wins = __ballot_sync(MSA_FULL_MASK, in_win);
        const bool ends = run < 32 && ((wins >> run) & 1u);
        if (state == 0) {
          if (lane < run) oc[i - lane] = 1;
          if (run > 0) pending = 0;
          i -= run;
          j -= run;
          if (ends) {
            const uint32_t src = __shfl_sync(MSA_FULL_MASK, code, run) & 3u;
            if (src == 0u) { ok = true; break; }
            state = src == 2u ? 1 : 2;
          }
        } else {
          const int n = run + (ends ? 1 : 0);  // a step that opens the gap ends it
          if (state == 1) {
            if (n > 0) pending = 0;
            i -= n;
          } else {
            pending += n;
            if (lane == 0 && n > 0) in[i] = (uint16_t)pending;
            j -= n;
          }
          if (ends) state = 0;
        }
      }
      if (i < 1 || j < 1) {  // the matrix's edge: H = 0
        ok = ok || state == 0;
        break;
      }
    }
    if (!ok && lane == 0) atomicOr(job.err, MSA_DERR_TRACE);
    const int i1 = bv > 0 ? i : 0, j1 = bv > 0 ? j : 0;
    const int e2 = bv > 0 ? i2 : 0, f2 = bv > 0 ? j2 : 0;
    // the flanks: the prefix right-aligned, the suffix left-aligned, surplus
    // residues in slots 0 and Lc
    const int kp = min(i1, j1);
    for (int t = lane; t < kp; t += 32) oc[i1 - t] = 1;
    const int a = Lc - e2, b = L - f2, ks = min(a, b);
    for (int t = lane + 1; t <= ks; t += 32) oc[e2 + t] = 1;
    __syncwarp();
    if (lane == 0) {
      // (the walk counts no E step at row 0, nor at the best cell's row: a cell
      // reached along its row scores less than one before it)
      if (j1 > i1) in[0] = (uint16_t)(j1 - i1);
      if (b > a) in[Lc] = (uint16_t)(b - a);
      int32_t *sg = job.seg + (size_t)orig * 5;
      sg[0] = bv; sg[1] = i1; sg[2] = j1; sg[3] = e2; sg[4] = f2;
      job.score[orig] = bv;
    }
  }
}

int few_warps(int Lc) { return std::min(kFewThreads / 32, (Lc + kStrip - 1) / kStrip); }

int few_smem(int K, int Lc, int maxlen) {
  return (K + 1) * round_up_int(Lc, kStrip) + round_up_int(maxlen, 16);
}

}  // namespace

size_t few_slot_codes(int Lc, int maxlen) { return (size_t)((Lc + kR - 1) / kR) * few_row_slots(maxlen); }

int few_grid(int K, int Lc, int maxlen, int n) {
  const int smem = few_smem(K, Lc, maxlen);
  int dev = 0, sms = 0, per_sm = 0, most = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (allow_smem((const void *)k_align_few, &most) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (smem > most) return 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_align_few, 32 * few_warps(Lc), smem);
  return (int)std::min<int64_t>(n, (int64_t)per_sm * std::max(sms, 1));
}

bool few_rounds(int Lc) { return (Lc + kStrip - 1) / kStrip > kFewThreads / 32; }

cudaError_t launch_align_few(const SeqSet &ss, const Scoring &sc, const FewJob &job, int Lc, int maxlen,
                             int grid, cudaStream_t st) {
  k_align_few<<<grid, 32 * few_warps(Lc), few_smem(sc.K, Lc, maxlen), st>>>(ss, sc, job);
  return cudaGetLastError();
}

// Microseconds of the alignment with its traceback, the launch aside, by
// k_align_few.  A step of a warp's strip measured 0.14 us alone on its
// scheduler and 0.088 us per warp where several share one (1 to 16 warps per
// SM, 80- to 5,000-residue centers), a walk 4 us and 0.02 us per residue, the
// profile 4 us and 2.3 ns per residue of the center.
double few_cost(int Lc, int n, double mean_len, int grid, int sms) {
  const int W = few_warps(Lc), nstrip = (Lc + kStrip - 1) / kStrip, rounds = (nstrip + W - 1) / W;
  const double steps = mean_len + 31 + kStep / 2;
  const double total = (rounds - 1) * std::max(steps + kStep, (double)W * kLag) + ((nstrip - 1) % W) * kLag + steps;
  const int ctas = std::max(1, std::min(n, grid));
  const double step = std::max(0.14, 0.088 * ctas * W / (4.0 * std::max(sms, 1)));
  const double walk = 4.0 + 0.02 * std::min((double)Lc, mean_len);
  return 4.0 + 0.0023 * Lc + std::ceil((double)n / ctas) * (total * step + walk);
}
