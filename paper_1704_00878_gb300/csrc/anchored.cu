// anchored.cu -- alignment of similar sequences to the center by anchors (the
// paper's trie path for similar nucleotides: the center's segments are
// indexed, matched segments of the other sequence are skipped and only the
// unmatched stretches are aligned).
//
// The center is cut into non-overlapping segments of k residues; their keys
// (k residues of ceil(log2 K) bits each) are sorted on the host and held in
// shared memory.  One warp per subject:
//   - the lanes roll the keys of the subject's k-mers over contiguous chunks;
//     a bit table of the segments' hashed keys turns almost every position
//     without a match away, the rest binary-search the keys, and every
//     (segment, position) match is collected;
//   - the matches are ordered by (segment, position) by counting per segment;
//   - the longest chain (increasing segment, sequence positions at least k
//     apart; a match's predecessor is the first compatible match of the
//     longest chains before it): the smallest end position of every chain
//     length grows with the length, so a match's length is one look at the
//     longest chain so far, or a warp-wide count when that one does not fit;
//   - the stretches between consecutive anchors are aligned globally (Gotoh,
//     W = open + (n-1) extend, traceback from the end: diagonal, then F, then
//     E; a gap extends only when strictly better): one lane per stretch of at
//     most 8 center residues, 32 stretches at a time; eight lanes (an
//     anti-diagonal wavefront) per stretch of at most 32; the whole warp for
//     taller ones.
// The flanks follow the local path's rule.  A subject with no match, more
// matches than the warp holds (the smallest power of two >= max(64, 2S)), or
// a stretch longer than kBoxSide on either side goes to the Smith-Waterman
// kernels instead.
// Bound by issue and the latency of a warp's serial steps (16 warps per SM, the
// match lists and workspaces fill shared memory).  50,000 subjects of 1,500
// nucleotides, k = 8 (127 matches, 41 stretches each): 6.6 ms with a binary
// search for every position, a bitonic sort, a chain recurrence over all
// earlier matches and one stretch at a time, 2.4 ms so.
#include <algorithm>
#include <climits>
#include <cstring>
#include <vector>

#include "ctx.cuh"
#include "dp_pass.cuh"

namespace msa_detail {
namespace {

constexpr int kAnchThreads = 256, kAnchWarps = kAnchThreads / 32;  // at most
constexpr int kBoxSide = 80;                         // longest stretch side
constexpr int kLaneCols = 24;                        // columns of a stretch that one lane aligns
constexpr int kLaneSort = 16;                        // matches of a segment that one lane orders
constexpr int kHashBits = 15;                        // bit table of the segments' keys
constexpr int kNeg = -(1 << 29);                      // stands for minus infinity
constexpr int kPosBits = 13;                          // match = segment << 13 | position

struct AnchJob {
  int center;                          // sorted index
  int nseg, k, bits;
  const unsigned long long *seg_key;   // sorted segment keys
  const int32_t *seg_id;               // the segment of each sorted key
  int cap;                             // matches a warp holds (power of two)
  uint16_t *ins;
  uint8_t *occ;
  int32_t *seg;
  int32_t *score;
  int32_t *fallback;                   // subjects (sorted index) left to the local path
  unsigned *nfallback;
  unsigned long long *counter;
};

// Per-warp workspace of the stretch aligner: one code byte per cell and two
// ping-pong rows (H and F of a pass's bottom row) for stretches of more than
// 32 center residues.
constexpr int kRowInts = 2 * (kBoxSide + 1);
constexpr int kStretchBytes = kBoxSide * kBoxSide + 2 * kRowInts * 4;

__device__ __forceinline__ int gap_cost(int len, int o, int e) { return -(o + (len - 1) * e); }

// Global affine alignment of the stretch c[0..lc) x x[0..lx) by the whole
// warp (center residue cb + i + 1 is c[i]); writes its columns to the row and
// returns its score (the same value in every lane).  Lanes hold center rows
// (32 per pass) and sweep the columns as an anti-diagonal wavefront: the cell
// above comes from the lane above by shuffle, the row above a pass from the
// workspace.  Gotoh with W_k = o + (k - 1) e, the edges charged from the
// stretch's corner; the codes (source 1 diagonal / 2 F / 3 E, ties in that
// order; E and F extend only when strictly better) go to shared memory and
// lane 0 walks them back from the end.
__device__ int stretch_align_warp(const uint8_t *__restrict__ c, int lc, const uint8_t *__restrict__ x,
                                  int lx, const int8_t *__restrict__ sM, int K, int o, int e, int cb,
                                  uint16_t *__restrict__ in, uint8_t *__restrict__ oc,
                                  uint8_t *__restrict__ work, int lane) {
  if (lc == 0 && lx == 0) return 0;
  if (lc == 0) {  // residues inserted before center residue cb + 1
    if (lane == 0) in[cb] = (uint16_t)lx;
    return gap_cost(lx, o, e);
  }
  if (lx == 0) return gap_cost(lc, o, e);  // center residues against gaps
  uint8_t *codes = work;
  int *rows = reinterpret_cast<int *>(work + kBoxSide * kBoxSide);
  int hlast = 0;
  const int npass = (lc + 31) / 32;
  for (int p = 0; p < npass; ++p) {
    const int i0 = 32 * p, R = min(32, lc - i0);
    const int *rin = rows + ((p + 1) & 1) * kRowInts;  // H, F of row i0 (pass p > 0)
    int *rout = rows + (p & 1) * kRowInts;
    const int i = i0 + lane + 1;  // this lane's row (1-based)
    const bool row_ok = lane < R;
    const int8_t *srow = sM + (row_ok ? c[i - 1] : 0) * K;
    int hs = 0, fs = kNeg, hl = 0, el = kNeg, hup_prev = 0;
    const int steps = lx + R - 1;
    for (int k = 0; k < steps; ++k) {
      int hup = __shfl_up_sync(MSA_FULL_MASK, hs, 1), fup = __shfl_up_sync(MSA_FULL_MASK, fs, 1);
      const int j = k - lane + 1;
      if (lane == 0 && j <= lx) {
        hup = p == 0 ? gap_cost(j, o, e) : rin[j];
        fup = p == 0 ? kNeg : rin[kBoxSide + 1 + j];
      }
      if (row_ok && j >= 1 && j <= lx) {
        int hdiag = hup_prev;
        if (j == 1) {
          hl = gap_cost(i, o, e);                         // H(i, 0)
          el = kNeg;
          hdiag = i == 1 ? 0 : gap_cost(i - 1, o, e);     // H(i - 1, 0)
        }
        const int eo = hl - o, ee = el - e, E = max(eo, ee);
        const int fo = hup - o, fe = fup - e, F = max(fo, fe);
        const int d = hdiag + srow[x[j - 1]];
        const int h = max(d, max(E, F));
        const int src = h == d ? 1 : (h == F ? 2 : 3);
        codes[(i - 1) * lx + (j - 1)] = (uint8_t)(src | ((ee > eo) << 2) | ((fe > fo) << 3));
        hs = h; fs = F; hl = h; el = E;
        if (lane == R - 1 && p + 1 < npass) { rout[j] = h; rout[kBoxSide + 1 + j] = F; }
        if (i == lc && j == lx) hlast = h;
      }
      hup_prev = hup;
    }
    __syncwarp();
  }
  const int score = __shfl_sync(MSA_FULL_MASK, hlast, (lc - 1) & 31);
  if (lane == 0) {
    int i = lc, j = lx, state = 0;  // 0 = H, 1 = F (center residue vs gap), 2 = E (inserted residue)
    int cnt = 0;                    // residues inserted at row i
    while (i > 0 || j > 0) {
      if (state == 0) {
        if (i == 0) state = 2;
        else if (j == 0) state = 1;
        else {
          const int src = codes[(i - 1) * lx + (j - 1)] & 3;
          if (src == 1) {
            oc[cb + i] = 1;
            if (cnt) in[cb + i] = (uint16_t)cnt;
            cnt = 0;
            --i;
            --j;
            continue;
          }
          state = src == 2 ? 1 : 2;
        }
      }
      if (state == 1) {
        const bool ext = j == 0 ? i > 1 : ((codes[(i - 1) * lx + (j - 1)] >> 3) & 1);
        if (cnt) in[cb + i] = (uint16_t)cnt;
        cnt = 0;
        --i;
        state = ext ? 1 : 0;
      } else {
        const bool ext = i == 0 ? j > 1 : ((codes[(i - 1) * lx + (j - 1)] >> 2) & 1);
        ++cnt;
        --j;
        state = ext ? 2 : 0;
      }
    }
    if (cnt) in[cb] = (uint16_t)cnt;
  }
  __syncwarp();
  return score;
}

// One cell of the stretches' recurrence (el, hl: E and H of the cell to the
// left; fup, hup: of the cell above; d: the diagonal's H plus the score): E, F,
// H and the 4-bit code.  Source 1 + a + b (1 diagonal, 2 F, 3 E), bits 2 and 3
// E and F extended: clamped differences of ordered values, put together by
// multiply-adds beside the integer pipe.
__device__ __forceinline__ uint32_t stretch_cell(int hl, int el, int hup, int fup, int d, int o, int e,
                                                 int &E, int &F, int &h) {
  const int eo = hl - o, fo = hup - o;
  E = max(eo, el - e);
  F = max(fo, fup - e);
  h = max(d, max(E, F));
  const int a = min(h - d, 1), b = min(h - F, a);
  return mad_lo((uint32_t)min(F - fo, 1), 8u, mad_lo((uint32_t)min(E - eo, 1), 4u, (uint32_t)(1 + a + b)));
}

// Global affine alignment of one stretch per active lane, c[0..lc) x
// x[0..lx) with lc <= 8 and lx <= kLaneCols, the recurrence and traceback of
// stretch_align_warp; every lane of the warp calls it.  Rows in registers,
// columns one after another, a column's codes in one word per lane.  Returns
// the lane's score (0 when inactive).
__device__ __forceinline__ int stretch_align_lane(bool active, const uint8_t *__restrict__ c, int lc,
                                  const uint8_t *__restrict__ x, int lx,
                                  const int8_t *__restrict__ sM, int K, int o, int e, int cb,
                                  uint16_t *__restrict__ in, uint8_t *__restrict__ oc,
                                  uint32_t *__restrict__ work, int lane) {
  constexpr int NR = 8;
  if (!active) lc = lx = 0;
  int hl[NR], el[NR], crow[NR];
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    crow[i] = i < lc ? (int)c[i] * K : 0;
    hl[i] = gap_cost(i + 1, o, e);  // H(i + 1, 0)
    el[i] = kNeg;
  }
  int score = 0, hcorner = 0;  // H(0, j - 1)
  for (int j = 1; j <= lx; ++j) {
    const int xj = x[j - 1];
    int hdiag = hcorner, hup = gap_cost(j, o, e), fup = kNeg;
    hcorner = hup;
    uint32_t w = 0;
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      int E, F, h;
      w = mad_lo(stretch_cell(hl[i], el[i], hup, fup, hdiag + sM[crow[i] + xj], o, e, E, F, h), 1u << (4 * i), w);
      hdiag = hl[i];
      hl[i] = h;
      el[i] = E;
      hup = h;
      fup = F;
      if (i + 1 == lc) score = h;
    }
    work[(j - 1) * 32 + lane] = w;
  }
  // (a lane reads back its own words)
  int i = lc, j = lx, state = 0, cnt = 0;
  while (i > 0 || j > 0) {
    if (i == 0) state = 2;
    else if (j == 0) state = 1;
    const uint32_t code = i > 0 && j > 0 ? work[(j - 1) * 32 + lane] >> (4 * (i - 1)) : 0u;
    if (state == 0) {
      const uint32_t src = code & 3u;
      if (src == 1u) {
        oc[cb + i] = 1;
        if (cnt) in[cb + i] = (uint16_t)cnt;
        cnt = 0;
        --i;
        --j;
        continue;
      }
      state = src == 2u ? 1 : 2;
    }
    if (state == 1) {
      const bool ext = j == 0 ? i > 1 : ((code >> 3) & 1u) != 0u;
      if (cnt) in[cb + i] = (uint16_t)cnt;
      cnt = 0;
      --i;
      state = ext ? 1 : 0;
    } else {
      const bool ext = i == 0 ? j > 1 : ((code >> 2) & 1u) != 0u;
      ++cnt;
      --j;
      state = ext ? 2 : 0;
    }
  }
  if (cnt) in[cb] = (uint16_t)cnt;  // i = 0
  return score;
}

// Four stretches at a time, one per group of eight lanes (lc <= 8 RPL, lx <=
// kBoxSide; every lane of the warp calls it, a group without a stretch with
// lc = lx = 0): RPL center rows per lane, an anti-diagonal wavefront over the
// group, a lane's codes of a step in one 16-bit word.  The group walks the
// codes back looking eight cells ahead along the path's direction.  Returns
// the score in the lane that holds row lc, 0 in the others.
template <int RPL>
__device__ __forceinline__ int stretch_align_group(const uint8_t *__restrict__ c, int lc,
                                   const uint8_t *__restrict__ x, int lx, const int8_t *__restrict__ sM,
                                   int K, int o, int e, int cb, uint16_t *__restrict__ in,
                                   uint8_t *__restrict__ oc, uint8_t *__restrict__ work, int lane) {
  static_assert(RPL <= 4, "a 16-bit word per lane and step");
  const int gl = lane & 7, grp = lane >> 3;
  uint16_t *codes = reinterpret_cast<uint16_t *>(work);                // [step][lane]
  uint8_t *sx = work + (kBoxSide + 7) * 64 + grp * kBoxSide;           // the group's residues
  for (int u = gl; u < lx; u += 8) sx[u] = x[u];
  const int i0 = gl * RPL;  // rows i0 + 1 .. i0 + RPL
  int hl[RPL], el[RPL], crow[RPL];
#pragma unroll
  for (int r = 0; r < RPL; ++r) {
    crow[r] = i0 + r < lc ? (int)c[i0 + r] * K : 0;
    hl[r] = gap_cost(i0 + r + 1, o, e);  // H(i, 0)
    el[r] = kNeg;
  }
  __syncwarp();
  const int steps = __reduce_max_sync(MSA_FULL_MASK, lx) + 7;
  int hbot = 0, fbot = kNeg, hprev = gl == 0 ? 0 : gap_cost(i0, o, e);  // H(i0, j - 1)
  int score = 0;
  for (int k = 0; k < steps; ++k) {
    int hup = __shfl_up_sync(MSA_FULL_MASK, hbot, 1), fup = __shfl_up_sync(MSA_FULL_MASK, fbot, 1);
    const int j = k - gl + 1;
    if (j < 1 || j > lx) continue;
    if (gl == 0) {
      hup = gap_cost(j, o, e);
      fup = kNeg;
    }
    int hdiag = hprev;
    hprev = hup;
    const int xj = sx[j - 1];
    uint32_t w = 0;
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
      int E, F, h;
      w = mad_lo(stretch_cell(hl[r], el[r], hup, fup, hdiag + sM[crow[r] + xj], o, e, E, F, h), 1u << (4 * r), w);
      hdiag = hl[r];
      hl[r] = h;
      el[r] = E;
      hup = h;
      fup = F;
      if (j == lx && i0 + r + 1 == lc) score = h;
    }
    hbot = hup;
    fbot = fup;
    codes[k * 32 + lane] = (uint16_t)w;
  }
  __syncwarp();
  int i = lc, j = lx, state = 0, cnt = 0;  // the same in a group's lanes; cnt: E steps at row i
  while (__any_sync(MSA_FULL_MASK, i > 0 && j > 0)) {
    const bool on = i > 0 && j > 0;
    const int ri = state == 2 ? i : i - gl, cj = state == 1 ? j : j - gl;
    const bool inside = on && ri >= 1 && cj >= 1;
    uint32_t code = 0;
    if (inside) {
      const int l = (ri - 1) / RPL;
      code = codes[(cj - 1 + l) * 32 + grp * 8 + l] >> (4 * ((ri - 1) % RPL));
    }
    const bool go = inside && (state == 0 ? (code & 3u) == 1u : ((code >> (state == 1 ? 3 : 2)) & 1u) != 0u);
    const unsigned stops = (~__ballot_sync(MSA_FULL_MASK, go) >> (8 * grp)) & 0xffu;
    const unsigned ins = (__ballot_sync(MSA_FULL_MASK, inside) >> (8 * grp)) & 0xffu;
    const int run = stops ? __ffs(stops) - 1 : 8;
    const bool ends = run < 8 && ((ins >> run) & 1u);
    const uint32_t src = __shfl_sync(MSA_FULL_MASK, code, grp * 8 + min(run, 7)) & 3u;
    if (!on) continue;
    if (state == 0) {
      if (gl < run) oc[cb + ri] = 1;
      if (run > 0) cnt = 0;
      i -= run;
      j -= run;
      if (ends) state = src == 2u ? 1 : 2;
    } else {
      const int n = run + (ends ? 1 : 0);
      if (state == 1) {
        if (n > 0) cnt = 0;
        i -= n;
      } else {
        cnt += n;
        if (gl == 0) in[cb + i] = (uint16_t)cnt;
        j -= n;
      }
      if (ends) state = 0;
    }
  }
  if (i == 0 && j > 0 && gl == 0) in[cb] = (uint16_t)j;
  __syncwarp();
  return score;
}

__device__ __forceinline__ uint32_t key_bit(unsigned long long key) {
  return (uint32_t)((key * 0x9e3779b97f4a7c15ull) >> (64 - kHashBits));
}
__device__ __forceinline__ uint32_t key_bit(uint32_t key) { return (key * 0x9e3779b1u) >> (32 - kHashBits); }

// Sorts v[0..n) by the whole warp: a bitonic network whose first step of every
// size compares mirrored positions, so that all comparisons are ascending and
// those that reach past n (a place that holds the largest value) do nothing.
__device__ void warp_sort(uint32_t *v, int n, int lane) {
  for (int size = 2; size < 2 * n; size <<= 1)
    for (int d = size >> 1; d > 0; d >>= 1) {
      const bool mirrored = d == size >> 1;
      for (int p = lane;; p += 32) {
        const int i = ((p & ~(d - 1)) << 1) | (p & (d - 1)), j = mirrored ? i ^ (size - 1) : i + d;
        if (i >= n) break;
        if (j >= n) continue;
        const uint32_t a = v[i], b = v[j];
        if (a > b) {
          v[i] = b;
          v[j] = a;
        }
      }
      __syncwarp();
    }
}

// Per-warp shared memory: `cap` sorted matches (4 bytes), three 16-bit arrays
// of cap entries, and an area that holds the unsorted matches and the
// segments' counts first and the stretch aligners' workspace later.
__host__ __device__ inline int anch_area(int cap) {
  const int m = cap * 6 + 32;
  return ((m > kStretchBytes ? m : kStretchBytes) + 15) & ~15;
}
__host__ __device__ inline int anch_warp_bytes(int cap) { return cap * 10 + anch_area(cap); }

// KEY: unsigned where a segment's key fits 32 bits, else unsigned long long.
template <class KEY>
__global__ void __launch_bounds__(kAnchThreads, 2) k_anchored(SeqSet ss, Scoring sc, AnchJob job,
                                                            const int32_t *__restrict__ perm) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int8_t sM[MSA_MAX_ALPHABET * MSA_MAX_ALPHABET];
  __shared__ uint32_t s_bits[(1 << kHashBits) / 32];
  __shared__ int s_nm[kAnchWarps], s_subj[kAnchWarps];
  const int K = sc.K, kk = job.k, S = job.nseg, NT = (int)blockDim.x;
  unsigned long long *skey = reinterpret_cast<unsigned long long *>(smem);
  int32_t *sid = reinterpret_cast<int32_t *>(skey + S);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char *mem = smem + (((size_t)S * 12 + 15) & ~(size_t)15) + (size_t)w * anch_warp_bytes(job.cap);
  uint8_t *work = mem;                                          // the area
  uint32_t *raw = reinterpret_cast<uint32_t *>(mem);            // unsorted matches
  int *segat = reinterpret_cast<int *>(raw + job.cap);          // counts, then ends, per segment
  uint32_t *mbuf = reinterpret_cast<uint32_t *>(mem + anch_area(job.cap));
  uint16_t *mlen = reinterpret_cast<uint16_t *>(mbuf + job.cap);  // chain length ending at a match
  uint16_t *minpos = mlen + job.cap;                              // [l - 1]: smallest end of length l
  uint16_t *first = minpos + job.cap;                             // [l - 1]: first match of length l
  for (int i = threadIdx.x; i < K * K; i += NT) sM[i] = sc.M[i];
  for (int i = threadIdx.x; i < (1 << kHashBits) / 32; i += NT) s_bits[i] = 0u;
  for (int i = threadIdx.x; i < S; i += NT) { skey[i] = job.seg_key[i]; sid[i] = job.seg_id[i]; }
  __syncthreads();
  for (int i = threadIdx.x; i < S; i += NT) {
    const uint32_t b = key_bit((KEY)skey[i]);
    atomicOr(&s_bits[b >> 5], 1u << (b & 31));
  }
  __syncthreads();
  const KEY mask = job.bits * kk >= 8 * (int)sizeof(KEY) ? ~(KEY)0 : (((KEY)1 << (job.bits * kk)) - (KEY)1);
  const uint32_t pmask = (1u << kPosBits) - 1;
  const int Lc = ss.len[job.center];
  const uint8_t *rc = ss.res + ss.pstart[job.center];
  for (;;) {
    __syncwarp();  // every lane is done with the last subject's shared state
    if (lane == 0) {
      s_subj[w] = (int)atomicAdd(job.counter, 1ull);
      s_nm[w] = 0;
    }
    for (int s = lane; s < S; s += 32) segat[s] = 0;
    __syncwarp();
    const int kx = s_subj[w];
    if (kx >= ss.n) break;
    const int Ls = ss.len[kx];
    const uint8_t *x = ss.res + ss.pstart[kx];
    // (a) every match of a center segment: the lanes roll the keys over
    // contiguous chunks (of k-mer ends, eight residues per load); positions
    // whose key's bit is set are listed and then searched for, all lanes at once
    {
      uint16_t *hits = minpos;  // 2 cap entries (and `first`)
      int nhit = 0;
      auto search = [&]() {
        __syncwarp();
        for (int i = lane; i < nhit; i += 32) {
          const int p = hits[i];
          unsigned long long key = 0ull;
          for (int u = 0; u < kk; ++u) key = (key << job.bits) | x[p + u];
          int lo = 0, hi = S;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (skey[mid] < key) lo = mid + 1; else hi = mid;
          }
          for (int q = lo; q < S && skey[q] == key; ++q) {
            const int slot = atomicAdd(&s_nm[w], 1);
            if (slot < job.cap) {
              raw[slot] = ((uint32_t)sid[q] << kPosBits) | (uint32_t)p;
              atomicAdd(&segat[sid[q]], 1);
            }
          }
        }
        __syncwarp();
        nhit = 0;
      };
      const int chunk = ((Ls + 31) / 32 + 7) & ~7, e0 = lane * chunk, e1 = min(Ls, e0 + chunk);
      KEY key = 0;
      if (e0 < e1)
        for (int u = max(0, e0 - kk + 1); u < e0; ++u) key = (key << job.bits) | x[u];
      const unsigned below = (1u << lane) - 1u;
      uint2 nxt = e0 < e1 ? *reinterpret_cast<const uint2 *>(x + e0) : make_uint2(0u, 0u);
      for (int c = 0; c < chunk; c += 8) {
        const uint2 v = nxt;
        const int eb = e0 + c;
        if (c + 8 < chunk && eb + 8 < e1) nxt = *reinterpret_cast<const uint2 *>(x + eb + 8);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          key = ((key << job.bits) | (((u < 4 ? v.x : v.y) >> (8 * (u & 3))) & 0xffu)) & mask;
          const uint32_t bit = key_bit(key);
          const bool hit = eb + u < e1 && eb + u >= kk - 1 && ((s_bits[bit >> 5] >> (bit & 31)) & 1u);
          const unsigned who = __ballot_sync(MSA_FULL_MASK, hit);
          if (who == 0u) continue;
          if (hit) hits[nhit + __popc(who & below)] = (uint16_t)(eb + u - kk + 1);
          nhit += __popc(who);
          if (nhit + 32 > 2 * job.cap) search();
        }
      }
      search();
    }
    const int M = s_nm[w];
    if (M == 0 || M > job.cap) {  // no anchor, or more matches than the warp holds
      if (lane == 0) {
        const unsigned slot = atomicAdd(job.nfallback, 1u);
        job.fallback[slot] = kx;
      }
      continue;
    }
    // (b) order the matches by (segment, position): starts by a scan of the
    // counts, then a segment's few matches sorted in place by one lane, the many
    // matches of a repeat by the warp (one lane's insertions are quadratic: 20,000
    // subjects with 208 and 338 matches of one segment 4.1 and 9.9 ms by one lane,
    // 0.70 and 1.02 by the warp)
    {
      const int per = (S + 31) / 32, s0 = min(S, lane * per), s1 = min(S, s0 + per);
      int sum = 0;
      for (int s = s0; s < s1; ++s) sum += segat[s];
      int incl = sum;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(MSA_FULL_MASK, incl, d);
        if (lane >= d) incl += v;
      }
      int at = incl - sum;
      for (int s = s0; s < s1; ++s) {
        const int n = segat[s];
        segat[s] = at;
        at += n;
      }
      __syncwarp();
      for (int i = lane; i < M; i += 32) {
        const uint32_t v = raw[i];
        mbuf[atomicAdd(&segat[v >> kPosBits], 1)] = v;
      }
      __syncwarp();
      for (int sb = 0; sb < S; sb += 32) {  // segat[s] is now the end of segment s
        const int s = sb + lane, end = s < S ? segat[s] : 0, b = s < S && s > 0 ? segat[s - 1] : 0;
        const bool many = end - b > kLaneSort;
        for (int i = b + 1; i < end && !many; ++i) {
          const uint32_t v = mbuf[i];
          int j = i;
          for (; j > b && mbuf[j - 1] > v; --j) mbuf[j] = mbuf[j - 1];
          mbuf[j] = v;
        }
        for (unsigned left = __ballot_sync(MSA_FULL_MASK, many); left; left &= left - 1) {
          const int l = __ffs(left) - 1, from = __shfl_sync(MSA_FULL_MASK, b, l);
          warp_sort(mbuf + from, __shfl_sync(MSA_FULL_MASK, end, l) - from, lane);
        }
      }
      __syncwarp();
    }
    // (c) longest chain.  A run of matches, each in a later segment than the
    // one before and fitting behind it, extends the longest chain one by one:
    // 32 at a time.  Any other match is taken with its segment's (they do not
    // chain with one another: all their lengths first, then the lengths'
    // smallest ends).
    int cur = 0, top = 0;  // the longest chain so far and its smallest end position
    for (int m = 0; m < M;) {
      {
        const uint32_t v = m + lane < M ? mbuf[m + lane] : 0xffffffffu;
        const uint32_t after = m + lane + 1 < M ? mbuf[m + lane + 1] : 0xffffffffu;
        const uint32_t before = __shfl_up_sync(MSA_FULL_MASK, v, 1);
        const int pos = (int)(v & pmask);
        const bool alone = m + lane < M && (after >> kPosBits) != (v >> kPosBits);
        const bool fits = lane == 0 ? cur == 0 || top + kk <= pos
                                    : (before >> kPosBits) != (v >> kPosBits) && (int)(before & pmask) + kk <= pos;
        const unsigned stop = ~__ballot_sync(MSA_FULL_MASK, alone && fits);
        const int run = stop ? __ffs(stop) - 1 : 32;
        if (run > 0) {
          if (lane < run) {
            mlen[m + lane] = (uint16_t)(cur + lane + 1);
            minpos[cur + lane] = (uint16_t)pos;
            first[cur + lane] = (uint16_t)(m + lane);
          }
          cur += run;
          top = __shfl_sync(MSA_FULL_MASK, pos, run - 1);
          m += run;
          __syncwarp();
          continue;
        }
      }
      const uint32_t sm = mbuf[m] >> kPosBits;
      int ge = m + 1;
      while (ge < M && (mbuf[ge] >> kPosBits) == sm) ++ge;
      const int cur0 = cur, top0 = top;
      for (int g = m; g < ge; ++g) {
        const int pos = (int)(mbuf[g] & pmask);
        int l = cur0;
        if (cur0 > 0 && top0 + kk > pos) {  // lengths whose smallest end fits: a prefix
          l = 0;
          for (int b = 0; b < cur0; b += 32) {
            const int t = b + lane;
            const unsigned fit = __ballot_sync(MSA_FULL_MASK, t < cur0 && (int)minpos[t] + kk <= pos);
            l += __popc(fit);
            if (fit != MSA_FULL_MASK) break;
          }
        }
        if (lane == 0) mlen[g] = (uint16_t)(l + 1);
      }
      __syncwarp();
      for (int g = m; g < ge; ++g) {
        const int pos = (int)(mbuf[g] & pmask), len = mlen[g];
        if (len > cur) {
          cur = len;
          top = pos;
          if (lane == 0) { minpos[len - 1] = (uint16_t)pos; first[len - 1] = (uint16_t)g; }
        } else {
          if (len == cur) top = min(top, pos);
          if (lane == 0 && pos < minpos[len - 1]) minpos[len - 1] = (uint16_t)pos;
        }
        __syncwarp();
      }
      m = ge;
    }
    // the chain (match indices, in order) into minpos[0..T), from its end: the
    // first match of the longest chains, then each predecessor -- the first
    // match of the length below that fits.  While the chain goes through the
    // first matches of their lengths, 32 steps at a time.
    const int T = cur;
    uint16_t *chain = minpos;
    {
      int t = T - 1, m = first[T - 1];
      __syncwarp();
      for (;;) {
        if (lane == 0) chain[t] = (uint16_t)m;
        if (t == 0) break;
        const uint32_t v = mbuf[m];
        auto fits = [&](int q, uint32_t behind) {
          const uint32_t u = mbuf[q];
          return (u >> kPosBits) < (behind >> kPosBits) && (int)(u & pmask) + kk <= (int)(behind & pmask);
        };
        if (m == first[t]) {
          const int tl = t - lane;  // this lane's step: from first[tl] to first[tl - 1]
          const bool ok = tl > 0 && fits(first[tl - 1], mbuf[first[tl]]);
          const unsigned stop = ~__ballot_sync(MSA_FULL_MASK, ok);
          const int run = stop ? __ffs(stop) - 1 : 32;
          if (run > 0) {
            if (lane < run) chain[tl - 1] = first[tl - 1];
            t -= run;
            m = first[t];
            continue;
          }
        }
        int q = first[t - 1];
        if (!fits(q, v)) {
          for (int b = q + 1; b < m; b += 32) {
            const int u = b + lane;
            const unsigned hit = __ballot_sync(MSA_FULL_MASK, u < m && (int)mlen[u] == t && fits(u, v));
            if (hit) { q = b + __ffs(hit) - 1; break; }
          }
        }
        m = q;
        --t;
      }
      __syncwarp();
    }
    auto anchor_s = [&](int t) { return (int)(mbuf[chain[t]] >> kPosBits); };
    auto anchor_p = [&](int t) { return (int)(mbuf[chain[t]] & pmask); };
    // (d) stretches too long send the subject to the local path
    bool big = false;
    for (int t = lane; t + 1 < T; t += 32) {
      const int lc = anchor_s(t + 1) * kk - (anchor_s(t) * kk + kk);
      const int lx = anchor_p(t + 1) - (anchor_p(t) + kk);
      big |= lc > kBoxSide || lx > kBoxSide;
    }
    if (__any_sync(MSA_FULL_MASK, big)) {
      if (lane == 0) {
        const unsigned slot = atomicAdd(job.nfallback, 1u);
        job.fallback[slot] = kx;
      }
      continue;
    }
    // (e) anchors, stretches, flanks: the row of this subject
    const int orig = perm[kx];
    uint16_t *in = job.ins + (size_t)orig * (Lc + 1);
    uint8_t *oc = job.occ + (size_t)orig * (Lc + 1);
    int score = 0;  // this lane's share
    for (int t = lane; t < T; t += 32) {
      const int ca = anchor_s(t) * kk, xa = anchor_p(t);
      for (int u = 0; u < kk; ++u) {
        oc[ca + u + 1] = 1;
        score += sM[rc[ca + u] * K + x[xa + u]];
      }
    }
    // stretches with residues on both sides: up to 8 center residues in the
    // front of a list, up to 16 from its back, the others in another (the
    // arrays of the chain's search are done with)
    uint16_t *list = mlen, *tall = first;
    int nsmall = 0, nmid = 0, ntall = 0;
    for (int t0 = 0; t0 + 1 < T; t0 += 32) {
      const int t = t0 + lane;
      int kind = 0;
      if (t + 1 < T) {
        const int cb = anchor_s(t) * kk + kk;
        const int lc = anchor_s(t + 1) * kk - cb, lx = anchor_p(t + 1) - (anchor_p(t) + kk);
        if (lc > 0 && lx > 0) {
          kind = lc <= 8 && lx <= kLaneCols ? 1 : lc <= 16 ? 2 : 3;
        } else if (lx > 0) {  // residues inserted before center residue cb + 1
          in[cb] = (uint16_t)lx;
          score += gap_cost(lx, sc.o, sc.e);
        } else if (lc > 0) {  // center residues against gaps
          score += gap_cost(lc, sc.o, sc.e);
        }
      }
      const unsigned a = __ballot_sync(MSA_FULL_MASK, kind == 1), b = __ballot_sync(MSA_FULL_MASK, kind == 2),
                     c = __ballot_sync(MSA_FULL_MASK, kind == 3);
      const unsigned below = (1u << lane) - 1u;
      if (kind == 1) list[nsmall + __popc(a & below)] = (uint16_t)t;
      if (kind == 2) list[job.cap - 1 - nmid - __popc(b & below)] = (uint16_t)t;
      if (kind == 3) tall[ntall + __popc(c & below)] = (uint16_t)t;
      nsmall += __popc(a);
      nmid += __popc(b);
      ntall += __popc(c);
    }
    __syncwarp();
    // stretch t: its center residues and their count, its residues and count
    auto c0_of = [&](int t) { return anchor_s(t) * kk + kk; };
    auto lc_of = [&](int t) { return anchor_s(t + 1) * kk - c0_of(t); };
    auto x0_of = [&](int t) { return anchor_p(t) + kk; };
    auto lx_of = [&](int t) { return anchor_p(t + 1) - x0_of(t); };
    for (int i = 0; i < nsmall; i += 32) {
      const bool on = i + lane < nsmall;
      const int t = on ? list[i + lane] : 0;
      const int cb = on ? c0_of(t) : 0;
      score += stretch_align_lane(on, rc + cb, on ? lc_of(t) : 0, on ? x + x0_of(t) : x, on ? lx_of(t) : 0, sM, K,
                                  sc.o, sc.e, cb, in, oc, reinterpret_cast<uint32_t *>(work), lane);
    }
    __syncwarp();
    for (int i = 0; i < nmid; i += 4) {
      const bool on = i + (lane >> 3) < nmid;
      const int t = on ? list[job.cap - 1 - i - (lane >> 3)] : 0;
      const int cb = on ? c0_of(t) : 0;
      score += stretch_align_group<2>(rc + cb, on ? lc_of(t) : 0, on ? x + x0_of(t) : x, on ? lx_of(t) : 0, sM, K,
                                      sc.o, sc.e, cb, in, oc, work, lane);
    }
    for (int i = 0; i < ntall; i += 4) {
      const int t = i + (lane >> 3) < ntall ? tall[i + (lane >> 3)] : -1;
      const bool on = t >= 0 && lc_of(t) <= 32;
      const int cb = on ? c0_of(t) : 0;
      score += stretch_align_group<4>(rc + cb, on ? lc_of(t) : 0, on ? x + x0_of(t) : x, on ? lx_of(t) : 0, sM, K,
                                      sc.o, sc.e, cb, in, oc, work, lane);
      // taller ones by the whole warp
      for (unsigned left = __ballot_sync(MSA_FULL_MASK, t >= 0 && !on && (lane & 7) == 0); left; left &= left - 1) {
        const int tt = __shfl_sync(MSA_FULL_MASK, t, __ffs(left) - 1);
        const int v = stretch_align_warp(rc + c0_of(tt), lc_of(tt), x + x0_of(tt), lx_of(tt), sM, K, sc.o, sc.e,
                                         c0_of(tt), in, oc, work, lane);
        if (lane == 0) score += v;
      }
    }
    score = (int)__reduce_add_sync(MSA_FULL_MASK, (unsigned)score);
    {
      const int i1 = anchor_s(0) * kk, j1 = anchor_p(0);
      const int i2 = anchor_s(T - 1) * kk + kk, j2 = anchor_p(T - 1) + kk;
      const int kp = min(i1, j1);
      for (int t = lane; t < kp; t += 32) oc[i1 - t] = 1;
      const int a = Lc - i2, b = Ls - j2, ks = min(a, b);
      for (int t = lane + 1; t <= ks; t += 32) oc[i2 + t] = 1;
      if (lane == 0) {
        if (j1 > i1) in[0] = (uint16_t)(j1 - i1);
        if (b > a) in[Lc] = (uint16_t)(b - a);
        int32_t *sg = job.seg + (size_t)orig * 5;
        sg[0] = score; sg[1] = i1; sg[2] = j1; sg[3] = i2; sg[4] = j2;
        job.score[orig] = score;
      }
    }
    __syncwarp();
  }
}

int anchored_smem(int nseg, int cap, int warps) {
  return ((nseg * 12 + 15) & ~15) + warps * anch_warp_bytes(cap);
}

constexpr int kAnchStatic = 6 * 1024;  // the kernel's static shared memory, rounded up

// shared memory by which the segments of a center are accepted (12 bytes per
// segment, eight warps with 8 bytes per match and a stretch workspace each)
int nseg_limit(int nseg, int cap) {
  return nseg * 12 + (nseg & 1) * 4 + kAnchWarps * cap * 8 + kAnchWarps * kStretchBytes;
}

// The local path (Smith-Waterman fill with codes, traceback) for a list of
// subjects (sorted indices, ascending length) over a view of the set whose
// last entry is the center; rows land at their input indices.
int align_subset_local(msa_ctx *ctx, int kc, const std::vector<int32_t> &subj, float &ms) {
  const int nv = (int)subj.size() + 1;
  std::vector<int64_t> vstart(nv);
  std::vector<int32_t> vlen(nv), vperm(nv);
  for (int v = 0; v + 1 < nv; ++v) {
    vstart[v] = ctx->pstart[subj[v]];
    vlen[v] = ctx->len_sorted[subj[v]];
    vperm[v] = ctx->perm[subj[v]];
  }
  vstart[nv - 1] = ctx->pstart[kc];
  vlen[nv - 1] = ctx->len_sorted[kc];
  vperm[nv - 1] = ctx->perm[kc];
  const int Lc = vlen[nv - 1];
  const bool packed = align_packed(ctx, Lc);
  const int R = kCodesR, G = align_lanes(ctx, Lc, packed);
  const int npass = (Lc + G * R - 1) / (G * R);
  std::vector<int64_t> offs(nv, 0);
  int64_t acc = 0;
  for (int v = 0; v + 1 < nv; ++v) { offs[v] = acc; acc += (int64_t)code_words(vlen[v], Lc, G) * 8; }
  DevBuf vs, vl, vp, vo;
  auto cleanup = [&]() { for (DevBuf *b : {&vs, &vl, &vp, &vo}) release(ctx, *b); };
  int rc = [&]() -> int {
    TRY(ensure(ctx, vs, sizeof(int64_t) * nv));
    TRY(ensure(ctx, vl, sizeof(int32_t) * nv));
    TRY(ensure(ctx, vp, sizeof(int32_t) * nv));
    TRY(ensure(ctx, vo, sizeof(int64_t) * nv));
    CK(cudaMemcpyAsync(vs.p, vstart.data(), sizeof(int64_t) * nv, cudaMemcpyHostToDevice, ctx->st));
    CK(cudaMemcpyAsync(vl.p, vlen.data(), sizeof(int32_t) * nv, cudaMemcpyHostToDevice, ctx->st));
    CK(cudaMemcpyAsync(vp.p, vperm.data(), sizeof(int32_t) * nv, cudaMemcpyHostToDevice, ctx->st));
    CK(cudaMemcpyAsync(vo.p, offs.data(), sizeof(int64_t) * nv, cudaMemcpyHostToDevice, ctx->st));
    const SeqSet vss{P<uint8_t>(ctx->res), P<int64_t>(vs), P<int32_t>(vl), nv};
    double total = 0.0;
    int vmax = 0, few = 0;
    for (int v = 0; v + 1 < nv; ++v) {
      total += vlen[v];
      vmax = std::max(vmax, vlen[v]);
    }
    if (align_few_wins(ctx, Lc, nv - 1, total / (nv - 1), vmax, &few)) {
      cudaEvent_t e0 = ctx->ev[2 * ST_TRACE], e1 = ctx->ev[2 * ST_TRACE + 1];
      CK(cudaEventRecord(e0, ctx->st));
      TRY(align_few(ctx, vss, nv - 1, nv - 1, P<int32_t>(vp), Lc, vmax, few));
      CK(cudaEventRecord(e1, ctx->st));
      CK(cudaStreamSynchronize(ctx->st));
      float t = 0.f;
      if (cudaEventElapsedTime(&t, e0, e1) == cudaSuccess) ms += t;
      return MSA_OK;
    }
    TRY(ensure(ctx, ctx->codes, (size_t)std::max<int64_t>(acc, 8)));
    TRY(ensure(ctx, ctx->best, sizeof(unsigned long long) * nv));
    const Scoring sc = scoring(ctx);
    const int smem = codes_smem_bytes(ctx->K, npass * G * R);
    const int cta = align_cta(ctx, G, packed);
    const int grid = codes_grid(G, packed, smem, cta);
    if (npass > 1)
      TRY(ensure(ctx, ctx->scratch, (size_t)grid * (codes_threads(packed, cta) / G) * 2 * ctx->maxlen * sizeof(int2)));
    CK(cudaMemsetAsync(ctx->dcounter, 0, sizeof(unsigned long long), ctx->st));
    CodesJob job;
    job.center = nv - 1;
    job.sb = 0;
    job.se = nv - 1;
    job.code_off = P<int64_t>(vo);
    job.codes = P<uint8_t>(ctx->codes);
    job.best = P<unsigned long long>(ctx->best);
    job.npass = npass;
    job.counter = ctx->dcounter;
    job.scratch = P<int2>(ctx->scratch);
    job.scratch_cols = ctx->maxlen;
    cudaEvent_t e0 = ctx->ev[2 * ST_TRACE], e1 = ctx->ev[2 * ST_TRACE + 1];
    CK(cudaEventRecord(e0, ctx->st));
    CK((++ctx->launches, launch_codes)(G, packed, vss, sc, job, grid, ctx->st, true, cta));
    CK((++ctx->launches, launch_traceback)(P<uint8_t>(ctx->codes), P<int64_t>(vo),
                                           P<unsigned long long>(ctx->best), 0, nv - 1,
                                           P<int32_t>(vl), P<int32_t>(vp), vss.res, vss.pstart,
                                           nv - 1, sc.M, sc.K, sc.o, sc.e, Lc, G,
                                           P<uint16_t>(ctx->ins), P<uint8_t>(ctx->occ),
                                           P<int32_t>(ctx->seg), P<int32_t>(ctx->score),
                                           ctx->derr, ctx->st, nullptr, nullptr, nullptr, nullptr,
                                           0u, 0));
    CK(cudaEventRecord(e1, ctx->st));
    CK(cudaStreamSynchronize(ctx->st));
    float t = 0.f;
    if (cudaEventElapsedTime(&t, e0, e1) == cudaSuccess) ms += t;
    return MSA_OK;
  }();
  cleanup();
  return rc;
}

}  // namespace
}  // namespace msa_detail

using namespace msa_detail;

extern "C" int msa_align_anchored(msa_ctx *ctx, int64_t center, int32_t k, int32_t *scores_out,
                                  int64_t *fallback_out) {
  if (!ctx) return MSA_EINVAL;
  if (ctx->n == 0) return fail(ctx, MSA_ESTATE, "no sequences loaded");
  if (center < 0 || center >= ctx->n) return fail(ctx, MSA_EINVAL, "center index out of range");
  int bits = 1;
  while ((1 << bits) < ctx->K) ++bits;
  if (k < 1 || k * bits > 64) return fail(ctx, MSA_EINVAL, "segment length %d outside 1..%d", k, 64 / bits);
  TRY(set_device(ctx));
  const int n = ctx->n;
  const int kc = ctx->inv[center];
  const int Lc = ctx->len_sorted[kc];
  if (Lc >= (1 << 13) || ctx->maxlen >= (1 << 13))
    return fail(ctx, MSA_ERANGE, "anchored path holds sequences below 8192 residues");
  ctx->aligned = ctx->merged = false;
  ctx->center = center;
  ctx->Lc = Lc;
  // the center's segment keys, sorted (host: one pass over Lc residues)
  const int S = Lc / k;
  std::vector<uint8_t> cres(Lc);
  CK(cudaMemcpyAsync(cres.data(), P<uint8_t>(ctx->res) + ctx->pstart[kc], Lc, cudaMemcpyDeviceToHost, ctx->st));
  CK(cudaStreamSynchronize(ctx->st));
  std::vector<std::pair<unsigned long long, int32_t>> segs(S);
  for (int s = 0; s < S; ++s) {
    unsigned long long key = 0ull;
    for (int u = 0; u < k; ++u) key = (key << bits) | cres[(size_t)s * k + u];
    segs[s] = {key, s};
  }
  std::sort(segs.begin(), segs.end());
  std::vector<unsigned long long> keys(S);
  std::vector<int32_t> ids(S);
  for (int s = 0; s < S; ++s) { keys[s] = segs[s].first; ids[s] = segs[s].second; }
  // matches a warp holds: the smallest power of two >= max(64, 2 S) (more
  // send the sequence to the local path); it must fit shared memory
  int cap = 64;
  while (cap < 2 * S) cap <<= 1;
  int dev_smem = 0;
  cudaDeviceGetAttribute(&dev_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->dev);
  // eight warps per CTA, fewer where their match lists would not fit
  int warps = kAnchWarps;
  while (warps > 1 && anchored_smem(S, cap, warps) + kAnchStatic > dev_smem) warps /= 2;
  const int smem = anchored_smem(S, cap, warps);
  if (nseg_limit(S, cap) + 2048 > dev_smem || smem + kAnchStatic > dev_smem)
    return fail(ctx, MSA_ERANGE, "%d center segments of k = %d need more shared memory", S, k);
  const size_t row = (size_t)Lc + 1;
  TRY(ensure(ctx, ctx->ins, sizeof(uint16_t) * row * n));
  TRY(ensure(ctx, ctx->occ, row * n));
  TRY(ensure(ctx, ctx->seg, sizeof(int32_t) * 5 * n));
  TRY(ensure(ctx, ctx->score, sizeof(int32_t) * n));
  DevBuf dk, di, df, dn;
  auto cleanup = [&]() { for (DevBuf *b : {&dk, &di, &df, &dn}) release(ctx, *b); };
  int rc = [&]() -> int {
    TRY(ensure(ctx, dk, sizeof(unsigned long long) * std::max(S, 1)));
    TRY(ensure(ctx, di, sizeof(int32_t) * std::max(S, 1)));
    TRY(ensure(ctx, df, sizeof(int32_t) * n));
    TRY(ensure(ctx, dn, sizeof(unsigned)));
    if (S > 0) {
      CK(cudaMemcpyAsync(dk.p, keys.data(), sizeof(unsigned long long) * S, cudaMemcpyHostToDevice, ctx->st));
      CK(cudaMemcpyAsync(di.p, ids.data(), sizeof(int32_t) * S, cudaMemcpyHostToDevice, ctx->st));
    }
    CK(cudaMemsetAsync(ctx->ins.p, 0, sizeof(uint16_t) * row * n, ctx->st));
    CK(cudaMemsetAsync(ctx->occ.p, 0, row * n, ctx->st));
    CK(cudaMemsetAsync(dn.p, 0, sizeof(unsigned), ctx->st));
    CK(cudaMemsetAsync(ctx->dcounter, 0, sizeof(unsigned long long), ctx->st));
    CK(cudaMemsetAsync(ctx->derr, 0, 2 * sizeof(unsigned), ctx->st));
    AnchJob job;
    job.center = kc;
    job.nseg = S;
    job.k = k;
    job.bits = bits;
    job.seg_key = P<unsigned long long>(dk);
    job.seg_id = P<int32_t>(di);
    job.cap = cap;
    job.ins = P<uint16_t>(ctx->ins);
    job.occ = P<uint8_t>(ctx->occ);
    job.seg = P<int32_t>(ctx->seg);
    job.score = P<int32_t>(ctx->score);
    job.fallback = P<int32_t>(df);
    job.nfallback = P<unsigned>(dn);
    job.counter = ctx->dcounter;
    auto fn = bits * k <= 32 ? k_anchored<uint32_t> : k_anchored<unsigned long long>;
    if (smem + kAnchStatic > 48 * 1024)
      CK(allow_smem((const void *)fn));
    int per_sm = 0, sms = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * warps, smem));
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->dev);
    const int grid = std::max(1, per_sm) * std::max(1, sms);
    stage_begin(ctx, ST_ALIGN);
    ++ctx->launches;
    fn<<<grid, 32 * warps, smem, ctx->st>>>(seqset(ctx), scoring(ctx), job, P<int32_t>(ctx->d_perm));
    CK(cudaGetLastError());
    stage_end(ctx, ST_ALIGN);
    unsigned nf = 0;
    CK(cudaMemcpyAsync(&nf, dn.p, sizeof(unsigned), cudaMemcpyDeviceToHost, ctx->st));
    CK(cudaStreamSynchronize(ctx->st));
    stage_collect(ctx, ST_ALIGN);
    float ms_local = 0.f;
    if (nf > 0) {
      std::vector<int32_t> fb(nf);
      CK(cudaMemcpyAsync(fb.data(), df.p, sizeof(int32_t) * nf, cudaMemcpyDeviceToHost, ctx->st));
      CK(cudaStreamSynchronize(ctx->st));
      std::sort(fb.begin(), fb.end());  // sorted positions ascend in length
      // chunks whose codes fit the budget
      const int G = align_lanes(ctx, Lc, align_packed(ctx, Lc));
      size_t budget = std::max<size_t>(ctx->codes_budget, code_words(ctx->maxlen, Lc, G) * 8);
      size_t acc = 0;
      std::vector<int32_t> part;
      for (size_t x = 0; x <= fb.size(); ++x) {
        const size_t sz = x < fb.size() ? code_words(ctx->len_sorted[fb[x]], Lc, G) * 8 : 0;
        if (x == fb.size() || (acc + sz > budget && !part.empty())) {
          if (!part.empty()) TRY(align_subset_local(ctx, kc, part, ms_local));
          part.clear();
          acc = 0;
          if (x == fb.size()) break;
        }
        part.push_back(fb[x]);
        acc += sz;
      }
    }
    ctx->stage_ms[ST_ALIGN_K] = ctx->stage_ms[ST_ALIGN];
    ctx->stage_ms[ST_TRACE] = ms_local;
    int64_t cells = 0;  // the local path's cells only (the anchored ones are not a full DP)
    if (fallback_out) *fallback_out = (int64_t)nf;
    ctx->cells[1] = cells;
    TRY(check_derr(ctx));
    if (scores_out) {
      CK(cudaMemcpyAsync(scores_out, ctx->score.p, sizeof(int32_t) * n, cudaMemcpyDefault, ctx->st));
      CK(cudaStreamSynchronize(ctx->st));
    }
    ctx->aligned = true;
    return MSA_OK;
  }();
  cleanup();
  return rc;
}
