// tree.cu -- the neighbour-joining tree over the MSA (the paper's section on
// NJ trees, Figure 4, citing Saitou and Nei): fixed-point p-distances between
// the merged rows, then neighbour joining on those integers.
//
// Distances: the rows become bit planes of their symbol indices (32 columns
// per word), a CTA takes a 64 x 64 tile of row pairs and combines the planes
// with three-input logic operations (k_planes, k_pdist).
//
// Neighbour joining: the matrix stays on the device (int32 -- every entry and
// joined distance within 2^30, else ERANGE -- positions in ascending slot
// order); one launch of a thread-block cluster runs the joins until half of the
// positions are left (k_nj_joins), then the matrix is packed to the active ones; the
// last 128 positions run in one CTA.
#include <algorithm>
#include <climits>
#include <vector>

#include "ctx.cuh"

namespace msa_detail {
namespace {

constexpr int kTile = 64;        // rows per side of a distance tile
constexpr int kPlaneWords = 15;  // 32-column words staged per step
constexpr int kSlab = 16384;     // rows whose planes are held at once
constexpr long long kDScale = 1LL << 20;
constexpr long long kDLimit = 1LL << 30;  // |distance| bound of the joins (int32 matrix)
constexpr int kJoinCtas = 16;      // CTAs of a large matrix's joins: one cluster,
constexpr int kJoinCtasFew = 8;    // smaller where the device has no room for it
constexpr int kSoloRows = 128;     // a matrix of at most this many positions: one CTA
constexpr int kScanSeg = 512;      // columns of one warp task of a row scan: 16 per lane
constexpr int kScanTasks = 256;    // scan results held at once (a row has at most 128 segments)
constexpr int kJoinSmem = 215 * 1024;

// ---------------------------------------------------------------- distances
// Bit planes of the listed rows (list null: rows r0, r0 + 1, ...): per 32
// columns a word per bit of the symbol index and a word of residue flags
// (not '-').  lo = planes 0-3 (0-2 and the flags where three planes hold the
// alphabet), hi = plane 4 and the flags.  One warp per word, one ballot per
// plane; words past the row's columns are zero.
template <bool WIDE>
__global__ void __launch_bounds__(256) k_planes(const uint8_t *__restrict__ msa, int64_t W,
                                                const int32_t *__restrict__ list, int r0, int rows,
                                                int words, const uint8_t *__restrict__ lut, int K,
                                                uint4 *__restrict__ lo, uint2 *__restrict__ hi) {
  __shared__ uint8_t slut[256];
  slut[threadIdx.x] = lut[threadIdx.x];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5, total = (int64_t)rows * words;
  for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < total; x += warps) {
    const int i = (int)(x / words), w = (int)(x - (int64_t)i * words);
    const int row = list ? list[r0 + i] : r0 + i;
    const int64_t c = (int64_t)w * 32 + lane;
    const int s = c < W ? slut[msa[(size_t)row * W + c]] : K + 1;
    const bool res = s <= K;  // K + 1 is the gap
    const unsigned v = res ? (unsigned)s : 0u;
    unsigned p[5];
#pragma unroll
    for (int b = 0; b < (WIDE ? 5 : 3); ++b) p[b] = __ballot_sync(MSA_FULL_MASK, (v >> b) & 1u);
    const unsigned m = __ballot_sync(MSA_FULL_MASK, res);
    if (lane == 0) {
      if (WIDE) {
        lo[x] = make_uint4(p[0], p[1], p[2], p[3]);
        hi[x] = make_uint2(p[4], m);
      } else {
        lo[x] = make_uint4(p[0], p[1], p[2], m);
      }
    }
  }
}

// Tiles of 64 x 64 row pairs.  SYM: A and B are the same rows; D[a][b] and
// D[b][a] stored (ld columns); NEAREST (near not null): per row of A the
// smallest (distance << 32 | position in B) by an atomic minimum -- the
// nearest row of B, ties to its first position.  a0 / b0: list positions of
// the slabs' first rows.
struct PdistJob {
  const uint4 *loA, *loB;
  const uint2 *hiA, *hiB;
  int words;       // per row, a multiple of kPlaneWords
  int nA, nB;      // rows of the slabs
  int a0, b0;
  size_t ld;
  unsigned long long *near;
};

// Distances from the planes: per 32 columns of a pair one three-input logic
// operation per plane gathers the differing symbols, two mask them to the
// columns both rows have, and the bits of three words are added up by a
// carry-save step before they are counted.  About 20 lane operations per 32
// column pairs where comparing four letters per 32-bit word took 72: integer
// (ALU) bound either way.  4,000 rows x 7,200 columns measured 5.4 ms with
// byte comparisons (their unaligned byte staging included) and 1.07 ms with the
// planes, the planes' own pass included.
template <bool WIDE, class T>
__global__ void __launch_bounds__(256, 2) k_pdist(PdistJob job, T *__restrict__ D) {
  const int ta = blockIdx.y, tb = blockIdx.x;
  const bool sym = job.near == nullptr;
  if (sym && job.a0 + ta * kTile > job.b0 + tb * kTile) return;
  __shared__ __align__(16) uint4 sAl[kTile][kPlaneWords], sBl[kTile][kPlaneWords];
  __shared__ __align__(16) uint2 sAh[WIDE ? kTile : 1][kPlaneWords], sBh[WIDE ? kTile : 1][kPlaneWords];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int a0 = ta * kTile, b0 = tb * kTile;
  uint32_t comp[4][4] = {}, mism[4][4] = {};
  for (int w0 = 0; w0 < job.words; w0 += kPlaneWords) {
    __syncthreads();
    for (int idx = threadIdx.x; idx < kTile * kPlaneWords; idx += 256) {
      const int r = idx / kPlaneWords, w = idx - r * kPlaneWords;
      const size_t ga = (size_t)(a0 + r) * job.words + w0 + w, gb = (size_t)(b0 + r) * job.words + w0 + w;
      const bool va = a0 + r < job.nA, vb = b0 + r < job.nB;
      sAl[r][w] = va ? job.loA[ga] : make_uint4(0u, 0u, 0u, 0u);
      sBl[r][w] = vb ? job.loB[gb] : make_uint4(0u, 0u, 0u, 0u);
      if (WIDE) {
        sAh[r][w] = va ? job.hiA[ga] : make_uint2(0u, 0u);
        sBh[r][w] = vb ? job.hiB[gb] : make_uint2(0u, 0u);
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int w = 0; w < kPlaneWords; w += 3) {
#pragma unroll
      for (int ih = 0; ih < 4; ih += 2) {  // two rows of A at a time (registers)
        uint4 al[2][3];
        uint2 ah[2][3];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int u = 0; u < 3; ++u) {
            al[i][u] = sAl[ty + 16 * (ih + i)][w + u];
            if (WIDE) ah[i][u] = sAh[ty + 16 * (ih + i)][w + u];
          }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint4 bl[3];
          uint2 bh[3];
#pragma unroll
          for (int u = 0; u < 3; ++u) {
            bl[u] = sBl[tx + 16 * j][w + u];
            if (WIDE) bh[u] = sBh[tx + 16 * j][w + u];
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            uint32_t c[3], m[3];
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              uint32_t x = al[i][u].x ^ bl[u].x;
              x |= al[i][u].y ^ bl[u].y;
              x |= al[i][u].z ^ bl[u].z;
              if (WIDE) {
                x |= al[i][u].w ^ bl[u].w;
                x |= ah[i][u].x ^ bh[u].x;
                c[u] = ah[i][u].y & bh[u].y;
              } else {
                c[u] = al[i][u].w & bl[u].w;
              }
              m[u] = x & c[u];
            }
            // one bits of three words: popc(sum) + 2 popc(carry)
            comp[ih + i][j] += __popc(c[0] ^ c[1] ^ c[2]) +
                               2 * __popc((c[0] & c[1]) | (c[2] & (c[0] | c[1])));
            mism[ih + i][j] += __popc(m[0] ^ m[1] ^ m[2]) +
                               2 * __popc((m[0] & m[1]) | (m[2] & (m[0] | m[1])));
          }
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int la = a0 + ty + 16 * i;
    if (la >= job.nA) continue;
    const int a = job.a0 + la;
    unsigned long long nearest = ~0ull;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int lb = b0 + tx + 16 * j;
      if (lb >= job.nB) continue;
      const int b = job.b0 + lb;
      const long long d = comp[i][j] ? ((long long)mism[i][j] * kDScale) / comp[i][j] : kDScale;
      if (sym) {
        D[(size_t)a * job.ld + b] = (T)d;
        D[(size_t)b * job.ld + a] = (T)d;
      } else {
        const unsigned long long key = ((unsigned long long)d << 32) | (unsigned)b;
        nearest = key < nearest ? key : nearest;
      }
    }
    if (!sym && nearest != ~0ull) atomicMin(&job.near[a], nearest);
  }
}

// ---------------------------------------------------------------- joins
// The joins of a matrix of P active positions until m_stop of them are left,
// in one launch of one cluster of NB CTAs (one CTA where P is small).  A join
// is a chain of short dependent steps, so what bounds it is latency, and the
// design keeps one cluster barrier per join and few trips to memory:
//   - CTA c owns the positions k = c, c + NB, ...; every CTA keeps its own
//     copy of all row sums and updates it itself from rows x and y, so only
//     the CTAs' best pairs cross the barrier (through distributed shared
//     memory);
//   - the new node's row goes to a staging row (two, by join parity) that its
//     owner copies over row x during the next join, when no CTA reads the old
//     row any more; column x is written by each row's owner, the only one
//     that scans that row;
//   - a row is scanned (the smallest (m - 2) d(k, y) - r_y over y > k and the
//     second) only when it may hold a Q below every known one.  Each owned
//     row carries its best known partner, whose value is recomputed exactly
//     each join, and a lower bound of its other entries: the second smallest
//     after a scan, then moved each join by the least any entry can have
//     changed -- it loses d(k, y) <= dmax_k as m - 2 falls by one and gains
//     what r_y lost, at least the least loss of any active y; the new column's
//     entry takes the partner's place or lowers the bound.  Rows whose bound
//     exceeds the smallest Q of the pairs known (the CTAs' last best pairs)
//     hold no better or equal pair but their partner's.  The new row's own
//     minimum comes from the pass that computes it.
// Smallest Q first, then the smallest (x, y): a skipped row's other pairs are
// strictly worse than a known pair, so ties are decided exactly.  On 4,000
// protein rows the first thousand joins scan about 5 rows each.  NJ of
// 4,000 rows: 83.6 ms with one launch scanning every tile and one
// joining, 27.9 ms so (latency: about 7 us a join, half of it row scans).
struct NjPick {
  long long q;
  unsigned xy;  // x << 16 | y
  int d;
};
__device__ __forceinline__ bool pick_less(const NjPick &u, const NjPick &v) {
  return u.q < v.q || (u.q == v.q && u.xy < v.xy);
}
// smallest of the lanes' 64-bit values: the high halves first, then the low
// halves of the lanes that hold the smallest high half
__device__ __forceinline__ long long warp_min_ll(long long v) {
  const int hi = __reduce_min_sync(MSA_FULL_MASK, (int)(v >> 32));
  const unsigned lo = __reduce_min_sync(MSA_FULL_MASK, (int)(v >> 32) == hi ? (unsigned)v : 0xffffffffu);
  return (long long)(((unsigned long long)(unsigned)hi << 32) | lo);
}
__device__ __forceinline__ NjPick warp_min(const NjPick &p) {
  NjPick o;
  o.q = warp_min_ll(p.q);
  o.xy = __reduce_min_sync(MSA_FULL_MASK, p.q == o.q ? p.xy : 0xffffffffu);
  const unsigned who = __ballot_sync(MSA_FULL_MASK, p.q == o.q && p.xy == o.xy);
  o.d = __shfl_sync(MSA_FULL_MASK, p.d, __ffs(who) - 1);
  return o;
}
// sum of the lanes' 64-bit values (24-bit pieces, each below 2^31 over a warp)
__device__ __forceinline__ long long warp_sum_ll(long long v) {
  const unsigned a = __reduce_add_sync(MSA_FULL_MASK, (unsigned)(v & 0xffffff));
  const unsigned b = __reduce_add_sync(MSA_FULL_MASK, (unsigned)((v >> 24) & 0xffffff));
  const int c = __reduce_add_sync(MSA_FULL_MASK, (int)(v >> 48));
  return (long long)a + ((long long)b << 24) + ((long long)c << 48);
}

struct NjJob {
  int *D;                 // P x P
  int P, m_stop, t0, n;   // all P positions active; join t0 is the next one
  long long *r;           // row sums, written back at the end
  uint8_t *act;           // written at the end: active positions
  int *node;
  int *joins;
  long long *lengths;     // numerators of the branch lengths over 2 (m - 2)
  int *stage;             // 2 x P staging rows
  long long *rcopy;       // null: the row sums sit in shared memory, else grid x P
  unsigned *err;
};

__device__ __forceinline__ uint32_t cluster_addr(const void *p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(r)
               : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}

// the distance of a pair from its value v = f d - r_y: (v + r_y) / f has no
// remainder; an estimate within 2^8, then the remainder's quotient exactly
__device__ __forceinline__ int pair_distance(long long v, long long ry, int f, float inv) {
  v += ry;
  const int d = __float2int_rn((float)v * inv);
  return d + __float2int_rn((float)(v - (long long)f * d) * inv);
}

constexpr long long kNjHigh = 1LL << 60;     // bound of a row without a partner

// NB CTAs (a power of two: owner and index of a position are a mask and a
// shift) of NT threads.
template <int NB, int NT>
__global__ void __launch_bounds__(NT, 1) k_nj_joins(NjJob job) {
  extern __shared__ __align__(16) long long nj_smem[];
  constexpr int NW = NT / 32;
  static_assert(NW <= 32 && NB <= 32, "one lane per warp, one per CTA");
  __shared__ __align__(16) NjPick s_pick[2][NB];  // every CTA's best pair, by join parity
  __shared__ NjPick s_wpick[NW];
  __shared__ long long s_sum[NW], s_new[2][NW];
  __shared__ int s_min[NW], s_top[NW], s_nlist;
  __shared__ long long s_scan[2][kScanTasks];  // a scan task's smallest and second key, largest entry
  __shared__ int s_stop[kScanTasks];
  const int P = job.P, cta = NB > 1 ? (int)(blockIdx.x & (NB - 1)) : 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nown = (P - cta + NB - 1) / NB, cap = (P + NB - 1) / NB;
  long long *L = nj_smem;               // per owned row: lower bound of its entries but cy's
  long long *r = L + cap;
  int *cy, *cd, *dm, *list;
  unsigned *act;
  {
    long long *p = r;
    if (job.rcopy) r = job.rcopy + (size_t)cta * P;
    else p += P;
    cy = reinterpret_cast<int *>(p);    // the row's best known partner (-1 none), its distance,
    cd = cy + cap;                      // an upper bound of the row's distances, the rows to
    dm = cd + cap;                      // scan
    list = dm + cap;
    act = reinterpret_cast<unsigned *>(list + cap);
  }
  auto active = [&](int k) { return (act[k >> 5] >> (k & 31)) & 1u; };
  auto wants_scan = [&](int i) { list[atomicAdd(&s_nlist, 1)] = i; };
  // a row's partner, bound and largest entry from its smallest and second keys
  auto set_row = [&](int i, long long b1, long long b2, int top, int f) {
    L[i] = b2 == LLONG_MAX ? kNjHigh : b2 >> 16;
    cy[i] = -1;
    cd[i] = 0;
    dm[i] = 0;
    if (b1 != LLONG_MAX) {
      const int y = (int)(b1 & 0xffff);
      cy[i] = y;
      cd[i] = pair_distance(b1 >> 16, r[y], f, 1.f / (float)f);
      dm[i] = top;
    }
  };
  for (int k = tid; k < P; k += NT) r[k] = job.r[k];
  for (int w = tid; w < (P + 31) / 32; w += NT)
    act[w] = 32 * w + 32 <= P ? 0xffffffffu : (1u << (P - 32 * w)) - 1u;
  if (tid == 0) s_nlist = 0;
  __syncthreads();
  for (int i = tid; i < nown; i += NT) wants_scan(i);
  __syncthreads();
  if constexpr (NB > 1) {  // every CTA has started before any writes to its shared memory
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  int m = P, t = job.t0, xprev = -1, xcur = -1;
  int *stage_cur = job.stage, *stage_prev = job.stage + P;
  int parity = 0;
  const NjPick none{LLONG_MAX, 0xffffffffu, 0};
  for (;;) {
    const int f = m - 2;
    // the listed rows' minima anew
    const int nlist = s_nlist;
    const int nseg = (P + kScanSeg - 1) / kScanSeg, chunk = kScanTasks / nseg;
    for (int l0 = 0; l0 < nlist; l0 += chunk) {
      const int rows = min(chunk, nlist - l0);
      for (int task = warp; task < rows * nseg; task += NW) {
        const int at = task / nseg, y0 = (task - at * nseg) * kScanSeg;
        const int k = list[l0 + at] * NB + cta;
        long long best = LLONG_MAX, next = LLONG_MAX;  // the smallest (value << 16 | y), the second
        int top = INT_MIN;
        if (y0 + kScanSeg > k + 1) {
          const int *row = k == xcur ? stage_prev : job.D + (size_t)k * P;
          int dv[kScanSeg / 32];
          unsigned ok = 0;
#pragma unroll
          for (int u = 0; u < kScanSeg / 32; ++u) {
            const int y = y0 + 32 * u + lane;
            const bool v = y > k && y < P && ((act[(y0 >> 5) + u] >> lane) & 1u);
            ok |= (v ? 1u : 0u) << u;
            dv[u] = v ? __ldcg(row + y) : 0;
          }
#pragma unroll
          for (int u = 0; u < kScanSeg / 32; ++u) {
            if (!((ok >> u) & 1u)) continue;
            const int y = y0 + 32 * u + lane;
            const long long v = (((long long)f * dv[u] - r[y]) << 16) | (long long)y;
            top = max(top, dv[u]);
            next = min(next, max(best, v));
            best = min(best, v);
          }
          const long long wbest = warp_min_ll(best);
          next = warp_min_ll(best == wbest ? next : best);
          best = wbest;
          top = __reduce_max_sync(MSA_FULL_MASK, top);
        }
        if (lane == 0) {
          s_scan[0][task] = best;
          s_scan[1][task] = next;
          s_stop[task] = top;
        }
      }
      __syncthreads();
      for (int at = tid; at < rows; at += NT) {
        const int i = list[l0 + at];
        long long b1 = LLONG_MAX, b2 = LLONG_MAX;
        int top = INT_MIN;
        for (int w = at * nseg; w < (at + 1) * nseg; ++w) {
          b2 = min(min(b2, s_scan[1][w]), max(b1, s_scan[0][w]));
          b1 = min(b1, s_scan[0][w]);
          top = max(top, s_stop[w]);
        }
        set_row(i, b1, b2, top, f);
      }
      __syncthreads();
    }
    // this CTA's best pair among its rows' partners, to every CTA
    NjPick best = none;
    for (int i = tid; i < nown; i += NT) {
      const int k = i * NB + cta;
      if (cy[i] < 0 || !active(k)) continue;
      const NjPick p{(long long)f * cd[i] - r[cy[i]] - r[k], ((unsigned)k << 16) | (unsigned)cy[i], cd[i]};
      if (pick_less(p, best)) best = p;
    }
    best = warp_min(best);
    if (lane == 0) s_wpick[warp] = best;
    if (tid == 0) s_nlist = 0;
    __syncthreads();
    NjPick *slots = s_pick[parity];
    if constexpr (NB > 1) {
      if (warp == 0) {
        best = warp_min(lane < NW ? s_wpick[lane] : none);
        if (lane < NB)
          asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                           cluster_addr(slots + cta, (uint32_t)lane)),
                       "r"((unsigned)best.q), "r"((unsigned)((unsigned long long)best.q >> 32)),
                       "r"(best.xy), "r"((unsigned)best.d)
                       : "memory");
      }
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    // lane c: CTA c's pair (one CTA: warp c's)
    const NjPick mine = NB > 1 ? (lane < NB ? slots[lane] : none) : (lane < NW ? s_wpick[lane] : none);
    best = warp_min(mine);
    parity ^= 1;
    if (best.xy == 0xffffffffu) {  // no pair (distances beyond their bound)
      if (tid == 0) atomicOr(job.err, MSA_DERR_RANGE);
      break;
    }
    // the join of x < y: the branch lengths' numerators, the new node n + t in
    // position x, its distances floor((d(x,k) + d(y,k) - d(x,y)) / 2), the row
    // sums, y retired
    const int x = (int)(best.xy >> 16), y = (int)(best.xy & 0xffffu);
    const long long dxy = best.d;
    if (cta == 0 && tid == 0) {
      job.lengths[2 * t] = f * dxy + r[x] - r[y];
      job.lengths[2 * t + 1] = f * dxy - r[x] + r[y];
      job.joins[2 * t] = job.node[x];
      job.joins[2 * t + 1] = job.node[y];
      job.node[x] = job.n + t;
    }
    xprev = xcur;
    xcur = x;
    const int *rowx = x == xprev ? stage_prev : job.D + (size_t)x * P;
    const int *rowy = y == xprev ? stage_prev : job.D + (size_t)y * P;
    // the last new row takes its place in the matrix (its owner; nobody reads
    // that row of the matrix during this join)
    const bool settle = xprev >= 0 && (xprev & (NB - 1)) == cta && xprev != x && xprev != y;
    const bool ownx = (x & (NB - 1)) == cta;
    const int f2 = f - 1;
    long long sum = 0, nbest = LLONG_MAX, nnext = LLONG_MAX;
    int cmin = INT_MAX, ntop = INT_MIN, big = 0;
    // this thread's owned row: its entries of rows x and y, in flight early
    const int kown = tid * NB + cta;
    const int axown = kown < P ? __ldcg(rowx + kown) : 0, ayown = kown < P ? __ldcg(rowy + kown) : 0;
    constexpr int U = 8;  // entries in flight per thread: loads first, then stores
    for (int base = 0; base < P; base += U * NT) {
      int a[U], b[U];
      long long rk[U];
      unsigned on = 0;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (base + u * NT >= P) break;  // the same for every thread
        const int k = base + u * NT + tid;
        const bool in = k < P && ((act[k >> 5] >> lane) & 1u) && k != x && k != y;
        on |= (in ? 1u : 0u) << u;
        a[u] = in ? __ldcg(rowx + k) : 0;
        b[u] = in ? __ldcg(rowy + k) : 0;
        rk[u] = in ? r[k] : 0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (base + u * NT >= P) break;
        if (!((on >> u) & 1u)) continue;
        const int k = base + u * NT + tid;
        // (entries within 2^30: the new one and the loss are within 1.5 * 2^30)
        const long long both = (long long)a[u] + b[u];
        const int dn = (int)((both - dxy) >> 1), loss = (int)(both - dn);
        big = max(big, dn < 0 ? -dn : dn);
        sum += dn;
        cmin = min(cmin, loss);
        rk[u] -= loss;
        r[k] = rk[u];
        if (ownx) {
          stage_cur[k] = dn;
          if (k > x) {  // the new row's own minimum
            const long long v = (((long long)f2 * dn - rk[u]) << 16) | (long long)k;
            nnext = min(nnext, max(nbest, v));
            nbest = min(nbest, v);
            ntop = max(ntop, dn);
          }
        }
      }
    }
    if (settle)
      for (int k = tid; k < P; k += NT)
        if (k != x) job.D[(size_t)xprev * P + k] = __ldcg(stage_prev + k);
    if (big > (int)kDLimit) atomicOr(job.err, MSA_DERR_RANGE);
    sum = warp_sum_ll(sum);
    cmin = __reduce_min_sync(MSA_FULL_MASK, cmin);
    if (lane == 0) { s_sum[warp] = sum; s_min[warp] = cmin; }
    if (ownx) {
      const long long wbest = warp_min_ll(nbest);
      nnext = warp_min_ll(nbest == wbest ? nnext : nbest);
      ntop = __reduce_max_sync(MSA_FULL_MASK, ntop);
      if (lane == 0) { s_new[0][warp] = wbest; s_new[1][warp] = nnext; s_top[warp] = ntop; }
    }
    __syncthreads();
    --m;
    ++t;
    { int *z = stage_cur; stage_cur = stage_prev; stage_prev = z; }  // stage_prev: row x
    cmin = __reduce_min_sync(MSA_FULL_MASK, lane < NW ? s_min[lane] : INT_MAX);
    sum = warp_sum_ll(lane < NW ? s_sum[lane] : 0);
    if (tid == 0) {
      r[x] = sum;
      act[y >> 5] &= ~(1u << (y & 31));
    }
    // the smallest Q of the last best pairs that live on
    long long ub = LLONG_MAX;
    {
      const int pa = (int)(mine.xy >> 16), pb = (int)(mine.xy & 0xffffu);
      if (mine.xy != 0xffffffffu && pa != x && pa != y && pb != x && pb != y)
        ub = (long long)f2 * mine.d - r[pa] - r[pb];
    }
    ub = warp_min_ll(ub);
    // the owned rows' new entries, partners and bounds; those that may hold a
    // better pair (the settled row is complete: its copy came before the
    // barrier)
    for (int i = tid; i < nown; i += NT) {
      const int k = i * NB + cta;
      if (k == y || (k != x && !active(k))) continue;
      if (k == x) {
        long long b1 = LLONG_MAX, b2 = LLONG_MAX;
        int top = INT_MIN;
        for (int w = 0; w < NW; ++w) {
          b2 = min(min(b2, s_new[1][w]), max(b1, s_new[0][w]));
          b1 = min(b1, s_new[0][w]);
          top = max(top, s_top[w]);
        }
        if (f2 > 0) set_row(i, b1, b2, top, f2);
        continue;
      }
      const int ax = i == tid ? axown : __ldcg(rowx + k), ay = i == tid ? ayown : __ldcg(rowy + k);
      const int dn = (int)(((long long)ax + ay - dxy) >> 1);
      job.D[(size_t)k * P + x] = dn;
      long long Li = L[i] + ((long long)cmin - dm[i]);
      int cyi = cy[i], cdi = cd[i];
      if (cyi == y || cyi == x) cyi = -1;
      if (k < x) {  // the new entry: the best known pair, or part of the rest
        const long long v = (long long)f2 * dn - sum;
        const long long was = cyi >= 0 ? (long long)f2 * cdi - r[cyi] : LLONG_MAX;
        if (cyi >= 0) Li = min(Li, max(v, was));
        if (v < was) { cyi = x; cdi = dn; }
        dm[i] = max(dm[i], dn);
        cd[i] = cdi;
      }
      L[i] = Li;
      cy[i] = cyi;
      if (Li - r[k] <= ub) wants_scan(i);
    }
    __syncthreads();
    if (m <= job.m_stop) break;
  }
  __syncthreads();
  // the last new row into the matrix; CTA 0 hands the state back
  if (xcur >= 0 && (xcur & (NB - 1)) == cta)
    for (int k = tid; k < P; k += NT)
      if (k != xcur && active(k)) job.D[(size_t)xcur * P + k] = __ldcg(stage_prev + k);
  if (cta == 0)
    for (int k = tid; k < P; k += NT) {
      job.r[k] = r[k];
      job.act[k] = active(k) ? 1 : 0;
    }
  if constexpr (NB > 1) {  // nobody leaves while a pair may still arrive
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// Positions of the active entries, ascending (one CTA; P <= 65536).
__global__ void __launch_bounds__(1024) k_nj_index(const uint8_t *__restrict__ act, int P,
                                                   int *__restrict__ idx) {
  __shared__ int wsum[32];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int base = 0; base < P; base += blockDim.x) {
    const int k = base + threadIdx.x;
    const int a = k < P && act[k] ? 1 : 0;
    int incl = a;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(MSA_FULL_MASK, incl, d);
      if (lane >= d) incl += v;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
      int v = wsum[lane];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(MSA_FULL_MASK, v, d);
        if (lane >= d) v += u;
      }
      wsum[lane] = v;
    }
    __syncthreads();
    const int before = carry + (w > 0 ? wsum[w - 1] : 0) + incl - a;
    if (a) idx[before] = k;
    __syncthreads();
    if (threadIdx.x == 0) carry += wsum[31];
    __syncthreads();
  }
}

// The matrix, row sums and node ids packed to the m active positions.
__global__ void k_nj_pack(const int *__restrict__ D, int P, const long long *__restrict__ r,
                          const int *__restrict__ node, const int *__restrict__ idx, int m,
                          int *__restrict__ D2, long long *__restrict__ r2,
                          int *__restrict__ node2) {
  const int u = blockIdx.y;
  const int su = idx[u];
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < m; v += gridDim.x * blockDim.x)
    D2[(size_t)u * m + v] = D[(size_t)su * P + idx[v]];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    r2[u] = r[su];
    node2[u] = node[su];
  }
}

// The branch lengths from their numerators (join t of n rows had m = n - t
// active: over 2 (m - 2), one correctly rounded division), in place, and the
// root: the two active positions joined at the middle of their edge.
__global__ void k_nj_finish(const int *__restrict__ D, int P, const uint8_t *__restrict__ act,
                            const int *__restrict__ node, int n, int *__restrict__ joins,
                            double *__restrict__ lengths) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, last = n - 2;
  if (i < 2 * last) {
    const long long num = __double_as_longlong(lengths[i]);
    lengths[i] = (double)num / (double)(2 * (long long)(last - (i >> 1)));
  }
  if (i != 0) return;
  int a = -1, b = -1;
  for (int k = 0; k < P; ++k)
    if (act[k]) {
      if (a < 0) a = k;
      else { b = k; break; }
    }
  if (a < 0 || b < 0) return;
  const double half = (double)D[(size_t)a * P + b] / 2.0;
  joins[2 * last] = node[a];
  joins[2 * last + 1] = node[b];
  lengths[2 * last] = half;
  lengths[2 * last + 1] = half;
}

// The int64 matrix into the int32 one the joins work on; entries beyond the
// bound set the range error.
__global__ void k_nj_narrow(const long long *__restrict__ D64, size_t count, int *__restrict__ D,
                            unsigned *__restrict__ err) {
  bool bad = false;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    const long long v = D64[i];
    bad |= v > kDLimit || v < -kDLimit;
    D[i] = (int)v;
  }
  if (bad) atomicOr(err, MSA_DERR_RANGE);
}

// Row sums (one warp per row), node ids, every position active.
__global__ void k_nj_init(long long *__restrict__ r, const int *__restrict__ D, int n,
                          int *__restrict__ node, uint8_t *__restrict__ act) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  for (int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n; k += warps) {
    long long s = 0;
    for (int j = lane; j < n; j += 32) s += j == k ? 0 : D[(size_t)k * n + j];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(MSA_FULL_MASK, s, off);
    if (lane == 0) {
      r[k] = s;
      node[k] = k;
      act[k] = 1;
    }
  }
}

// Bit planes of a slab of listed rows.
struct Planes {
  uint4 *lo = nullptr;
  uint2 *hi = nullptr;  // more than seven letters
  int rows = 0;
};

// The planes of rows r0, r0 + 1, ... (of the list: device, null = all rows)
// into p's memory.
int make_planes(msa_ctx *ctx, Planes &p, const int32_t *list, int r0, int rows, int words) {
  const size_t cells = (size_t)rows * words;
  const int blocks = (int)std::min<size_t>((cells + 31) / 32, 1 << 14);  // four words per warp or more
  ++ctx->launches;
  auto fn = ctx->K > 7 ? k_planes<true> : k_planes<false>;
  fn<<<std::max(blocks, 1), 256, 0, ctx->st>>>(P<uint8_t>(ctx->msa), ctx->W, list, r0, rows, words,
                                               ctx->dSymLut, ctx->K, p.lo, p.hi);
  CK(cudaGetLastError());
  p.rows = rows;
  return MSA_OK;
}

// Distances of the rows ia[0..nA) (device list, null = rows 0..nA-1) against
// ib[0..nB): into the matrix D (near null: both lists the same, nA x nA, T =
// int or long long), or each row of A's nearest row of B into near.  The
// planes are held a slab of rows at a time, fewer where a device memory limit
// leaves less; where it leaves no room for them they take the place of the
// traceback codes, which nothing reads between two calls.
template <class T>
int distances(msa_ctx *ctx, const int32_t *ia, int nA, const int32_t *ib, int nB, T *D,
              unsigned long long *near) {
  const int words = (int)((ctx->W + 32 * kPlaneWords - 1) / (32 * kPlaneWords)) * kPlaneWords;
  const size_t row = (size_t)words * (sizeof(uint4) + (ctx->K > 7 ? sizeof(uint2) : 0));
  int slab = std::min(kSlab, (std::max(nA, nB) + kTile - 1) / kTile * kTile);
  auto bytes = [&](int rows) { return row * rows * (near || nA > rows ? 2 : 1); };  // one slab, or two
  DevBuf own;
  char *mem = nullptr;
  if (ctx->dev_limit) {
    const size_t left = ctx->dev_limit > ctx->dev_bytes ? ctx->dev_limit - ctx->dev_bytes : 0;
    while (slab > kTile && bytes(slab) + 256 > left) slab = std::max(kTile, slab / 2 / kTile * kTile);
    if (bytes(slab) + 256 > left) {
      int rows = std::min(slab, std::max(nA, nB));
      while (rows > 1 && bytes(rows) > ctx->codes.cap) rows /= 2;
      if (bytes(rows) <= ctx->codes.cap) {
        slab = rows;
        mem = P<char>(ctx->codes);
      }
    }
  }
  int rc = [&]() -> int {
    if (!mem) {
      TRY(ensure(ctx, own, bytes(slab)));
      mem = P<char>(own);
    }
    Planes pa, pb;
    // (both slabs' 16-byte words first, so that every plane is aligned)
    const size_t cells = (size_t)slab * words;
    pa.lo = reinterpret_cast<uint4 *>(mem);
    pb.lo = pa.lo + cells;
    pa.hi = reinterpret_cast<uint2 *>(pa.lo + bytes(slab) / row * words);
    pb.hi = pa.hi + cells;
    for (int a0 = 0; a0 < nA; a0 += slab) {
      const int ra = std::min(slab, nA - a0);
      TRY(make_planes(ctx, pa, ia, a0, ra, words));
      for (int b0 = near ? 0 : a0; b0 < nB; b0 += slab) {
        const int rb = std::min(slab, nB - b0);
        const bool same = !near && b0 == a0;
        if (!same && (nB > slab || pb.rows == 0)) TRY(make_planes(ctx, pb, ib, b0, rb, words));
        Planes &q = same ? pa : pb;
        PdistJob job{pa.lo, q.lo, pa.hi, q.hi, words, ra, rb, a0, b0, (size_t)nA, near};
        ++ctx->launches;
        auto fn = ctx->K > 7 ? k_pdist<true, T> : k_pdist<false, T>;
        fn<<<dim3((rb + kTile - 1) / kTile, (ra + kTile - 1) / kTile), 256, 0, ctx->st>>>(job, D);
        CK(cudaGetLastError());
      }
    }
    return MSA_OK;
  }();
  release(ctx, own);
  return rc;
}

// Per cluster c of the sample: the smallest (d(t, s) << 32 | s) over sample
// positions t in c and s outside it (the outgroup: the nearest sample row
// outside, ties to the smaller row).
__global__ void k_outgroups(const int *__restrict__ D, int m, const int32_t *__restrict__ cl,
                            unsigned long long *__restrict__ key) {
  const int t = blockIdx.y;
  const int c = cl[t];
  unsigned long long best = ~0ull;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < m; s += gridDim.x * blockDim.x)
    if (cl[s] != c) {
      const unsigned long long k = ((unsigned long long)D[(size_t)t * m + s] << 32) | (unsigned)s;
      best = k < best ? k : best;
    }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(MSA_FULL_MASK, best, off);
    best = o < best ? o : best;
  }
  if ((threadIdx.x & 31) == 0 && best != ~0ull) atomicMin(&key[c], best);
}

using join_fn = void (*)(NjJob);
static join_fn join_kernel(int ctas, int threads) {
  if (ctas == 1) return k_nj_joins<1, 256>;
  if (ctas == kJoinCtasFew)
    return threads == 256 ? k_nj_joins<kJoinCtasFew, 256>
         : threads == 512 ? k_nj_joins<kJoinCtasFew, 512> : k_nj_joins<kJoinCtasFew, 1024>;
  return threads == 256 ? k_nj_joins<kJoinCtas, 256>
       : threads == 512 ? k_nj_joins<kJoinCtas, 512> : k_nj_joins<kJoinCtas, 1024>;
}

// One launch of the joins of P positions.
struct JoinShape {
  int ctas, threads;
  bool rshared;  // the row sums fit shared memory
  size_t smem;
};
static JoinShape join_shape(int P, int ctas, int threads, bool sums_global) {
  JoinShape s{ctas, threads, false, 0};
  const size_t cap = (size_t)(P + ctas - 1) / ctas;
  s.smem = cap * (sizeof(long long) + 4 * sizeof(int)) + sizeof(unsigned) * (((size_t)P + 31) / 32);
  s.rshared = !sums_global && s.smem + sizeof(long long) * (size_t)P <= (size_t)kJoinSmem;
  if (s.rshared) s.smem += sizeof(long long) * (size_t)P;
  return s;
}

// Fills cfg and attr for a launch of s (attr must outlive the launch).
static cudaError_t join_config(const JoinShape &s, cudaStream_t st, cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr) {
  const void *fn = (const void *)join_kernel(s.ctas, s.threads);
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kJoinSmem);
  if (e == cudaSuccess && s.ctas > 8) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)s.ctas;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg = {};
  cfg.gridDim = dim3((unsigned)s.ctas);
  cfg.blockDim = dim3((unsigned)s.threads);
  cfg.dynamicSmemBytes = s.smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = s.ctas > 1 ? 1 : 0;
  return e;
}

// fewer threads make the block-wide steps of a join cheaper, more keep more of
// rows x and y in flight
static int join_threads(int P) { return P <= 1536 ? 256 : P <= 8192 ? 512 : 1024; }

// CTAs of the joins' cluster: 16 (not portable: a partition of the device, or a
// GPC with fewer SMs, may have no room for it), else 8, which every device of
// this architecture runs.  4,000 rows 30.7 ms with 16, 36.4 with 8; 10,000 139
// and 168.
static int join_ctas(int n) {
  const JoinShape s = join_shape(n, kJoinCtas, join_threads(n), false);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  int clusters = 0;
  if (join_config(s, nullptr, cfg, attr) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&clusters, (const void *)join_kernel(s.ctas, s.threads), &cfg) == cudaSuccess &&
      clusters > 0)
    return kJoinCtas;
  cudaGetLastError();
  return kJoinCtasFew;
}

// Row sums and the joins of the n x n int32 matrix in D1 (device; repacked in
// place of copies as positions retire).  derr must be clear.
int nj_device(msa_ctx *ctx, DevBuf &D1, int n, int32_t *joins_out, double *lengths_out) {
  if (n < 2) return MSA_OK;
  DevBuf D2, r, r2, node, node2, act, idx, joins, lengths, stage, rcopy;
  auto cleanup = [&]() {
    for (DevBuf *b : {&D2, &r, &r2, &node, &node2, &act, &idx, &joins, &lengths, &stage, &rcopy})
      release(ctx, *b);
  };
  int rc = [&]() -> int {
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->dev);
    TRY(ensure(ctx, r, sizeof(long long) * n));
    TRY(ensure(ctx, node, sizeof(int) * n));
    TRY(ensure(ctx, act, (size_t)n));
    TRY(ensure(ctx, idx, sizeof(int) * n));
    TRY(ensure(ctx, stage, sizeof(int) * 2 * (size_t)n));
    TRY(ensure(ctx, joins, sizeof(int) * 2 * (size_t)(n - 1)));
    TRY(ensure(ctx, lengths, sizeof(double) * 2 * (size_t)(n - 1)));
    ++ctx->launches;
    k_nj_init<<<std::max(1, sms) * 8, 256, 0, ctx->st>>>(P<long long>(r), P<int>(D1), n, P<int>(node),
                                                         P<uint8_t>(act));
    CK(cudaGetLastError());
    DevBuf *cD = &D1, *cR = &r, *cN = &node;
    DevBuf *oD = &D2, *oR = &r2, *oN = &node2;
    int Pn = n, t = 0;
    const int ctas = ctx->nj_ctas > 0 ? ctx->nj_ctas : n > kSoloRows ? join_ctas(n) : 1;
    while (Pn > 2) {
      // a large matrix until half of its positions are left, then packed
      const bool solo = Pn <= kSoloRows;
      const int stop = solo ? 2 : std::max(kSoloRows, Pn / 2), grid = solo ? 1 : ctas;
      const int threads = grid == 1 ? 256 : ctx->nj_threads > 0 ? ctx->nj_threads : join_threads(Pn);
      const JoinShape s = join_shape(Pn, grid, threads, ctx->nj_sums_global);
      if (s.smem > (size_t)kJoinSmem) return fail(ctx, MSA_ERANGE, "%d rows do not fit %d CTAs", Pn, grid);
      if (!s.rshared) TRY(ensure(ctx, rcopy, sizeof(long long) * (size_t)Pn * grid));
      NjJob job{P<int>(*cD), Pn, stop, t, n, P<long long>(*cR), P<uint8_t>(act), P<int>(*cN),
                P<int>(joins), P<long long>(lengths), P<int>(stage),
                s.rshared ? nullptr : P<long long>(rcopy), ctx->derr};
      ++ctx->launches;
      cudaLaunchConfig_t cfg;
      cudaLaunchAttribute attr;
      CK(join_config(s, ctx->st, cfg, attr));
      void *args[] = {&job};
      CK(cudaLaunchKernelExC(&cfg, (const void *)join_kernel(s.ctas, s.threads), args));
      t += Pn - stop;
      if (stop <= 2) break;
      const int m = stop;
      TRY(ensure(ctx, *oD, sizeof(int) * (size_t)m * m));
      TRY(ensure(ctx, *oR, sizeof(long long) * m));
      TRY(ensure(ctx, *oN, sizeof(int) * m));
      ctx->launches += 2;
      k_nj_index<<<1, 1024, 0, ctx->st>>>(P<uint8_t>(act), Pn, P<int>(idx));
      CK(cudaGetLastError());
      k_nj_pack<<<dim3((m + 255) / 256, m), 256, 0, ctx->st>>>(P<int>(*cD), Pn, P<long long>(*cR), P<int>(*cN),
                                                               P<int>(idx), m, P<int>(*oD),
                                                               P<long long>(*oR), P<int>(*oN));
      CK(cudaGetLastError());
      std::swap(cD, oD);
      std::swap(cR, oR);
      std::swap(cN, oN);
      Pn = m;
    }
    ++ctx->launches;
    k_nj_finish<<<(2 * n + 255) / 256, 256, 0, ctx->st>>>(P<int>(*cD), Pn, P<uint8_t>(act), P<int>(*cN), n,
                                                         P<int>(joins), P<double>(lengths));
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(joins_out, joins.p, sizeof(int) * 2 * (size_t)(n - 1), cudaMemcpyDefault,
                       ctx->st));
    CK(cudaMemcpyAsync(lengths_out, lengths.p, sizeof(double) * 2 * (size_t)(n - 1),
                       cudaMemcpyDefault, ctx->st));
    TRY(check_derr(ctx));
    return MSA_OK;
  }();
  cleanup();
  return rc;
}

// Neighbour joining of the merged rows idx[0..m) (device list, null = all):
// their distances into D (int32, m x m), then the joins on a copy of D where
// keep is set (the caller needs the distances), else on D itself.
int nj_rows(msa_ctx *ctx, const int32_t *idx, int m, DevBuf &D, bool keep, int32_t *joins_out,
            double *lengths_out) {
  TRY(ensure(ctx, D, sizeof(int) * (size_t)m * m));
  TRY(distances<int>(ctx, idx, m, idx, m, P<int>(D), nullptr));
  if (m < 2) return MSA_OK;
  CK(cudaMemsetAsync(ctx->derr, 0, 2 * sizeof(unsigned), ctx->st));
  if (!keep) return nj_device(ctx, D, m, joins_out, lengths_out);
  DevBuf C;
  int rc = [&]() -> int {
    TRY(ensure(ctx, C, sizeof(int) * (size_t)m * m));
    CK(cudaMemcpyAsync(C.p, D.p, sizeof(int) * (size_t)m * m, cudaMemcpyDeviceToDevice, ctx->st));
    return nj_device(ctx, C, m, joins_out, lengths_out);
  }();
  release(ctx, C);
  return rc;
}

// ---------------------------------------------------------------- clustered tree (host side)
// A rooted tree: kids[v] = its (child, length) pairs, none for a leaf.
using Kids = std::vector<std::vector<std::pair<int, double>>>;

// The unrooted tree of NJ joins over nleaf leaves (node nleaf + t for join t;
// the last join's two edges become one edge, its node unused).
static Kids unrooted(const std::vector<int32_t> &joins, const std::vector<double> &lengths, int nleaf) {
  const int T = nleaf - 1;
  Kids adj(2 * nleaf);
  auto link = [&](int a, int b, double l) { adj[a].push_back({b, l}); adj[b].push_back({a, l}); };
  for (int t = 0; t + 1 < T; ++t) {
    link(nleaf + t, joins[2 * t], lengths[2 * t]);
    link(nleaf + t, joins[2 * t + 1], lengths[2 * t + 1]);
  }
  link(joins[2 * (T - 1)], joins[2 * (T - 1) + 1], lengths[2 * (T - 1)] + lengths[2 * (T - 1) + 1]);
  return adj;
}

// The leaf farthest from src (distances summed along the path from src,
// ties to the smaller leaf) and each node's (parent, edge) toward src.
static int farthest(const Kids &adj, int src, int nleaf, double &dist_out,
                    std::vector<std::pair<int, double>> &par) {
  std::vector<double> dist(adj.size(), 0.0);
  std::vector<char> seen(adj.size(), 0);
  par.assign(adj.size(), {-1, 0.0});
  std::vector<int> stack = {src};
  seen[src] = 1;
  while (!stack.empty()) {
    const int v = stack.back();
    stack.pop_back();
    for (auto [w, l] : adj[v])
      if (!seen[w]) {
        seen[w] = 1;
        dist[w] = dist[v] + l;
        par[w] = {v, l};
        stack.push_back(w);
      }
  }
  int best = -1;
  for (int v = 0; v < nleaf; ++v)
    if (best < 0 || dist[v] > dist[best]) best = v;
  dist_out = dist[best];
  return best;
}

// Orient the unrooted adjacency away from `root`, skipping node `drop`.
static Kids orient(const Kids &adj, int root, int drop) {
  Kids kids(adj.size());
  std::vector<char> seen(adj.size(), 0);
  seen[root] = 1;
  if (drop >= 0) seen[drop] = 1;
  std::vector<int> stack = {root};
  while (!stack.empty()) {
    const int v = stack.back();
    stack.pop_back();
    for (auto [w, l] : adj[v])
      if (!seen[w]) {
        seen[w] = 1;
        kids[v].push_back({w, l});
        stack.push_back(w);
      }
  }
  return kids;
}

// The NJ tree rooted at the middle of its longest leaf-to-leaf path (see
// msa_nj_cluster_tree); the new root is node 2 nleaf - 2.
static Kids midpoint_rooted(const std::vector<int32_t> &joins, const std::vector<double> &lengths,
                            int nleaf, int &root) {
  Kids adj = unrooted(joins, lengths, nleaf);
  std::vector<std::pair<int, double>> par;
  double total = 0.0;
  const int a = farthest(adj, 0, nleaf, total, par);
  const int b = farthest(adj, a, nleaf, total, par);
  const double half = total / 2.0;
  int v = b;
  double walked = 0.0, l = 0.0;
  int u = -1;
  for (;;) {  // the last edge of the path at the latest (negative lengths)
    u = par[v].first;
    l = par[v].second;
    if (walked + l >= half || u == a) break;
    walked += l;
    v = u;
  }
  const double x = half - walked;
  auto drop_edge = [&](int p, int q) {
    auto &e = adj[p];
    e.erase(std::find_if(e.begin(), e.end(), [&](const std::pair<int, double> &z) { return z.first == q; }));
  };
  drop_edge(v, u);
  drop_edge(u, v);
  root = 2 * nleaf - 2;
  adj[root] = {{v, x}, {u, l - x}};
  adj[v].push_back({root, x});
  adj[u].push_back({root, l - x});
  return orient(adj, root, -1);
}

// Copy a rooted tree (leaf ids mapped to rows by name[]) into the arena.
static int graft(const Kids &kids, int root, const std::vector<int> &name, int nleaf, Kids &arena) {
  // iterative: children are copied before their parent
  std::vector<std::pair<int, int>> stack = {{root, 0}};
  std::vector<int> made(kids.size(), -1);
  while (!stack.empty()) {
    auto &[v, state] = stack.back();
    if (kids[v].empty()) {
      made[v] = name[v < nleaf ? v : 0];
      stack.pop_back();
      continue;
    }
    if (state == 0) {
      state = 1;
      const int vv = v;
      for (auto [w, l] : kids[vv]) stack.push_back({w, 0});
      continue;
    }
    const int id = (int)arena.size();
    arena.emplace_back();
    for (auto [w, l] : kids[v]) arena[id].push_back({made[w], l});
    made[v] = id;
    stack.pop_back();
  }
  return made[root];
}

int cluster_tree(msa_ctx *ctx, const std::vector<int32_t> &S, int cap, int32_t *joins_out,
                 double *lengths_out, int32_t *cluster_out) {
  const int n = ctx->n, m = (int)S.size();
  DevBuf dS, dS2, dlist, dnear, dcl, dkey;
  auto cleanup = [&]() { for (DevBuf *b : {&dS, &dS2, &dlist, &dnear, &dcl, &dkey}) release(ctx, *b); };
  int rc = [&]() -> int {
    // 1. the sample tree, midpoint-rooted
    TRY(ensure(ctx, dlist, sizeof(int32_t) * std::max(n, 1)));
    CK(cudaMemcpyAsync(dlist.p, S.data(), sizeof(int32_t) * m, cudaMemcpyHostToDevice, ctx->st));
    std::vector<int32_t> sj(2 * std::max(m - 1, 0));
    std::vector<double> sl(2 * std::max(m - 1, 0));
    TRY(nj_rows(ctx, P<int32_t>(dlist), m, dS, true, sj.data(), sl.data()));
    CK(cudaStreamSynchronize(ctx->st));
    Kids skids;
    int sroot = 0;
    if (m > 1) skids = midpoint_rooted(sj, sl, m, sroot);
    else skids.assign(1, {});
    // leaves under every node (post-order)
    const int nn = (int)skids.size();
    std::vector<int> nleaves(nn, 0), lowleaf(nn, INT_MAX);
    {
      std::vector<std::pair<int, int>> stack = {{sroot, 0}};
      while (!stack.empty()) {
        auto &[v, st] = stack.back();
        if (skids[v].empty()) { nleaves[v] = 1; lowleaf[v] = v; stack.pop_back(); continue; }
        if (st == 0) { st = 1; const int vv = v; for (auto [w, l] : skids[vv]) stack.push_back({w, 0}); continue; }
        for (auto [w, l] : skids[v]) { nleaves[v] += nleaves[w]; lowleaf[v] = std::min(lowleaf[v], lowleaf[w]); }
        stack.pop_back();
      }
    }
    // 2. the cut: split the subtree holding the most sample rows (ties: the
    // smaller node; the root is never tied) until none holds more than cap
    std::vector<int> cuts = {sroot};
    for (;;) {
      int bi = 0;
      for (int k = 1; k < (int)cuts.size(); ++k) {
        const int v = cuts[k], w = cuts[bi];
        if (nleaves[v] > nleaves[w] || (nleaves[v] == nleaves[w] && v < w)) bi = k;
      }
      const int big = cuts[bi];
      if (nleaves[big] <= cap) break;
      cuts.erase(cuts.begin() + bi);
      for (auto [w, l] : skids[big]) cuts.push_back(w);
    }
    std::sort(cuts.begin(), cuts.end(), [&](int x, int y) { return lowleaf[x] < lowleaf[y]; });
    const int q = (int)cuts.size();
    std::vector<int32_t> leaf_cl(m, 0);
    {
      std::vector<int> is_cut(nn, -1);
      for (int c = 0; c < q; ++c) is_cut[cuts[c]] = c;
      std::vector<std::pair<int, int>> stack = {{sroot, -1}};
      while (!stack.empty()) {
        auto [v, c] = stack.back();
        stack.pop_back();
        if (is_cut[v] >= 0) c = is_cut[v];
        if (skids[v].empty()) leaf_cl[v] = c;
        for (auto [w, l] : skids[v]) stack.push_back({w, c});
      }
    }
    // 3. labels: sample rows their own cluster, others their nearest sample row's
    std::vector<int32_t> cluster(n, -1);
    {
      TRY(ensure(ctx, dnear, sizeof(unsigned long long) * n));
      CK(cudaMemsetAsync(dnear.p, 0xff, sizeof(unsigned long long) * n, ctx->st));
      TRY(distances<int>(ctx, nullptr, n, P<int32_t>(dlist), m, nullptr, P<unsigned long long>(dnear)));
      std::vector<unsigned long long> near(n);
      CK(cudaMemcpyAsync(near.data(), dnear.p, sizeof(unsigned long long) * n, cudaMemcpyDeviceToHost, ctx->st));
      CK(cudaStreamSynchronize(ctx->st));
      for (int i = 0; i < n; ++i) cluster[i] = leaf_cl[(int)(near[i] & 0xffffffffu)];
      for (int l = 0; l < m; ++l) cluster[S[l]] = leaf_cl[l];
    }
    // 4. outgroups
    std::vector<int> outgroup(q, -1);
    if (q > 1) {
      TRY(ensure(ctx, dcl, sizeof(int32_t) * m));
      TRY(ensure(ctx, dkey, sizeof(unsigned long long) * q));
      CK(cudaMemcpyAsync(dcl.p, leaf_cl.data(), sizeof(int32_t) * m, cudaMemcpyHostToDevice, ctx->st));
      CK(cudaMemsetAsync(dkey.p, 0xff, sizeof(unsigned long long) * q, ctx->st));
      ++ctx->launches;
      k_outgroups<<<dim3((m + 255) / 256, m), 256, 0, ctx->st>>>(P<int>(dS), m, P<int32_t>(dcl),
                                                                 P<unsigned long long>(dkey));
      CK(cudaGetLastError());
      std::vector<unsigned long long> key(q);
      CK(cudaMemcpyAsync(key.data(), dkey.p, sizeof(unsigned long long) * q, cudaMemcpyDeviceToHost, ctx->st));
      CK(cudaStreamSynchronize(ctx->st));
      for (int c = 0; c < q; ++c) outgroup[c] = S[(int)(key[c] & 0xffffffffu)];
    }
    // 5. cluster trees into the arena (rows 0..n-1 are its leaves)
    Kids arena(n);
    std::vector<int> rows_of_cut(nn, -1);  // arena root of each cut's cluster tree
    std::vector<std::vector<int>> members(q);
    for (int i = 0; i < n; ++i) members[cluster[i]].push_back(i);
    for (int c = 0; c < q; ++c) {
      const std::vector<int> &R = members[c];
      if (R.size() == 1) { rows_of_cut[cuts[c]] = R[0]; continue; }
      std::vector<int> U = R;
      int opos = -1;
      if (q > 1) {
        U.push_back(outgroup[c]);
        std::sort(U.begin(), U.end());
        opos = (int)(std::lower_bound(U.begin(), U.end(), outgroup[c]) - U.begin());
      }
      const int u = (int)U.size();
      if (u > kMaxTreeRows) return fail(ctx, MSA_ERANGE, "a cluster of %d rows (at most %d)", u, kMaxTreeRows);
      std::vector<int32_t> U32(U.begin(), U.end());
      CK(cudaMemcpyAsync(dlist.p, U32.data(), sizeof(int32_t) * u, cudaMemcpyHostToDevice, ctx->st));
      std::vector<int32_t> cj(2 * (u - 1));
      std::vector<double> cl(2 * (u - 1));
      TRY(nj_rows(ctx, P<int32_t>(dlist), u, dS2, false, cj.data(), cl.data()));
      CK(cudaStreamSynchronize(ctx->st));
      Kids ck;
      int croot;
      if (q == 1) {  // the NJ tree as it is rooted
        ck.assign(2 * u - 1, {});
        for (int t = 0; t < u - 1; ++t)
          ck[u + t] = {{cj[2 * t], cl[2 * t]}, {cj[2 * t + 1], cl[2 * t + 1]}};
        croot = 2 * u - 2;
      } else {  // rooted where the outgroup joins, the outgroup removed
        const Kids adj = unrooted(cj, cl, u);
        croot = adj[opos][0].first;
        ck = orient(adj, croot, opos);
      }
      std::vector<int> name(U.begin(), U.end());
      rows_of_cut[cuts[c]] = graft(ck, croot, name, u, arena);
    }
    // 6. the sample tree above the cuts, the cluster trees below
    int root;
    if (q == 1) {
      root = rows_of_cut[cuts[0]];
    } else {
      std::vector<int> made(nn, -1);
      std::vector<std::pair<int, int>> stack = {{sroot, 0}};
      while (!stack.empty()) {
        auto &[v, st] = stack.back();
        if (rows_of_cut[v] >= 0) { made[v] = rows_of_cut[v]; stack.pop_back(); continue; }
        if (st == 0) { st = 1; const int vv = v; for (auto [w, l] : skids[vv]) stack.push_back({w, 0}); continue; }
        const int id = (int)arena.size();
        arena.emplace_back();
        for (auto [w, l] : skids[v]) arena[id].push_back({made[w], l});
        made[v] = id;
        stack.pop_back();
      }
      root = made[sroot];
    }
    // 7. post-order, children by their smallest row, internal nodes n, n+1, ...
    if (n > 1) {
      const int na = (int)arena.size();
      std::vector<int> low(na, INT_MAX), id(na, -1);
      for (int i = 0; i < n; ++i) low[i] = i, id[i] = i;
      for (int v = n; v < na; ++v)  // arena children are always made before their parent
        for (auto [w, l] : arena[v]) low[v] = std::min(low[v], low[w]);
      for (int v = n; v < na; ++v)
        std::sort(arena[v].begin(), arena[v].end(),
                  [&](const std::pair<int, double> &x, const std::pair<int, double> &y) {
                    return low[x.first] < low[y.first];
                  });
      int t = 0;
      std::vector<std::pair<int, int>> stack = {{root, 0}};
      while (!stack.empty()) {
        auto &top = stack.back();
        const int v = top.first;
        if (v < n) { stack.pop_back(); continue; }
        if (top.second == 0) {
          top.second = 1;
          const int c0 = arena[v][0].first, c1 = arena[v][1].first;
          stack.push_back({c1, 0});  // the first child is finished first
          stack.push_back({c0, 0});
          continue;
        }
        id[v] = n + t;
        joins_out[2 * t] = id[arena[v][0].first];
        joins_out[2 * t + 1] = id[arena[v][1].first];
        lengths_out[2 * t] = arena[v][0].second;
        lengths_out[2 * t + 1] = arena[v][1].second;
        ++t;
        stack.pop_back();
      }
    }
    if (cluster_out) std::copy(cluster.begin(), cluster.end(), cluster_out);
    return MSA_OK;
  }();
  cleanup();
  return rc;
}

}  // namespace
}  // namespace msa_detail

using namespace msa_detail;

int msa_tree_distances(msa_ctx *ctx, int64_t *dist_out) {
  if (!ctx || !dist_out) return MSA_EINVAL;
  TRY(set_device(ctx));
  DevBuf D;
  int rc = [&]() -> int {
    if (!ctx->merged) return fail(ctx, MSA_ESTATE, "merge the alignment first");
    const size_t n = ctx->n;
    TRY(ensure(ctx, D, sizeof(long long) * n * n));
    stage_begin(ctx, ST_TREE);
    TRY(distances<long long>(ctx, nullptr, ctx->n, nullptr, ctx->n, P<long long>(D), nullptr));
    stage_end(ctx, ST_TREE);
    CK(cudaMemcpyAsync(dist_out, D.p, sizeof(long long) * n * n, cudaMemcpyDefault, ctx->st));
    CK(cudaStreamSynchronize(ctx->st));
    stage_collect(ctx, ST_TREE);
    return MSA_OK;
  }();
  release(ctx, D);
  return rc;
}

int msa_nj(msa_ctx *ctx, const int64_t *dist, int64_t n, int32_t *joins_out, double *lengths_out) {
  if (!ctx || !dist || n < 1 || n > kMaxTreeRows || ((!joins_out || !lengths_out) && n > 1))
    return MSA_EINVAL;
  TRY(set_device(ctx));
  DevBuf D, D1;
  int rc = [&]() -> int {
    const size_t count = (size_t)n * n;
    TRY(ensure(ctx, D, sizeof(long long) * count));
    CK(cudaMemcpyAsync(D.p, dist, sizeof(long long) * count, cudaMemcpyDefault, ctx->st));
    stage_begin(ctx, ST_TREE);
    if (n > 1) {
      TRY(ensure(ctx, D1, sizeof(int) * count));
      CK(cudaMemsetAsync(ctx->derr, 0, 2 * sizeof(unsigned), ctx->st));
      ++ctx->launches;
      k_nj_narrow<<<1216, 256, 0, ctx->st>>>(P<long long>(D), count, P<int>(D1), ctx->derr);
      CK(cudaGetLastError());
      TRY(nj_device(ctx, D1, (int)n, joins_out, lengths_out));
    }
    stage_end(ctx, ST_TREE);
    CK(cudaStreamSynchronize(ctx->st));
    stage_collect(ctx, ST_TREE);
    return MSA_OK;
  }();
  release(ctx, D);
  release(ctx, D1);
  return rc;
}

int msa_debug_nj_shape(msa_ctx *ctx, int32_t ctas, int32_t threads, int32_t sums_global) {
  if (!ctx || (ctas != 0 && ctas != 1 && ctas != kJoinCtasFew && ctas != kJoinCtas)) return MSA_EINVAL;
  if (threads != 0 && threads != 256 && threads != 512 && threads != 1024) return MSA_EINVAL;
  ctx->nj_ctas = ctas;
  ctx->nj_threads = threads;
  ctx->nj_sums_global = sums_global != 0;
  return MSA_OK;
}

int msa_nj_tree(msa_ctx *ctx, int32_t *joins_out, double *lengths_out) {
  if (!ctx) return MSA_EINVAL;
  if (ctx->n > 1 && (!joins_out || !lengths_out)) return MSA_EINVAL;
  if (ctx->n > kMaxTreeRows) return fail(ctx, MSA_ERANGE, "more than %d sequences", kMaxTreeRows);
  TRY(set_device(ctx));
  DevBuf D;
  int rc = [&]() -> int {
    if (!ctx->merged) return fail(ctx, MSA_ESTATE, "merge the alignment first");
    stage_begin(ctx, ST_TREE);
    TRY(nj_rows(ctx, nullptr, ctx->n, D, false, joins_out, lengths_out));
    stage_end(ctx, ST_TREE);
    CK(cudaStreamSynchronize(ctx->st));
    stage_collect(ctx, ST_TREE);
    return MSA_OK;
  }();
  release(ctx, D);
  return rc;
}

int msa_nj_cluster_tree(msa_ctx *ctx, const int64_t *sample, int64_t nsample, int32_t cap,
                        int32_t *joins_out, double *lengths_out, int32_t *cluster_out) {
  if (!ctx || !sample || nsample < 1 || cap < 1) return MSA_EINVAL;
  if (ctx->n > 1 && (!joins_out || !lengths_out)) return MSA_EINVAL;
  if (!ctx->merged) return fail(ctx, MSA_ESTATE, "merge the alignment first");
  std::vector<int32_t> S;
  S.reserve(nsample);
  for (int64_t k = 0; k < nsample; ++k) {
    if (sample[k] < 0 || sample[k] >= ctx->n) return fail(ctx, MSA_EINVAL, "sample row out of range");
    S.push_back((int32_t)sample[k]);
  }
  std::sort(S.begin(), S.end());
  S.erase(std::unique(S.begin(), S.end()), S.end());
  if ((int64_t)S.size() > kMaxTreeRows) return fail(ctx, MSA_ERANGE, "a sample of more than %d rows", kMaxTreeRows);
  TRY(set_device(ctx));
  std::vector<int32_t> joins(2 * (size_t)std::max(ctx->n - 1, 0));
  std::vector<double> lengths(joins.size());
  std::vector<int32_t> cluster(ctx->n);
  stage_begin(ctx, ST_TREE);
  TRY(cluster_tree(ctx, S, cap, joins.data(), lengths.data(), cluster.data()));
  stage_end(ctx, ST_TREE);
  CK(cudaStreamSynchronize(ctx->st));
  stage_collect(ctx, ST_TREE);
  if (!joins.empty()) {
    CK(cudaMemcpyAsync(joins_out, joins.data(), sizeof(int32_t) * joins.size(), cudaMemcpyDefault, ctx->st));
    CK(cudaMemcpyAsync(lengths_out, lengths.data(), sizeof(double) * lengths.size(), cudaMemcpyDefault, ctx->st));
  }
  if (cluster_out)
    CK(cudaMemcpyAsync(cluster_out, cluster.data(), sizeof(int32_t) * cluster.size(), cudaMemcpyDefault, ctx->st));
  CK(cudaStreamSynchronize(ctx->st));
  return MSA_OK;
}
