// Widest paths, all pairs (Sect. 2.1 definition; Sect. 4 "straightforward
// algorithm" computing p(a, b) for every pair), as a blocked Floyd-Warshall
// in the (max, min) semiring.
//
// Edge weights are winning votes, w[i][j] = d[i][j] if d[i][j] > d[j][i]
// else 0. They are packed into a zero-padded square workspace W (int16 when
// every count fits in 15 bits, else int32) whose rows and columns follow a
// relabeling of the candidates: candidates with at least one outgoing edge
// first, strongest first (most outgoing edges, or most ballots), then those
// without edges in id order. The closure commutes with relabeling, and rows
// without edges stay zero, so their tiles are never touched. The order
// among the warm candidates puts like widths into the same 64 x 64 tiles: a
// majority graph is close to an order, so below the diagonal most tiles are
// zero, and above it a tile's smallest entry soon reaches what a further
// pivot block could offer, which lets most tile updates be skipped (below).
//
// Only the candidates with edges (the "warm" ones, nw of them) need work:
// rows of cold candidates are zero in W and in p. W holds the warm rows only
// (padded to whole tiles), over all relabeled columns; warm columns come
// first. The closure has two parts:
//   * the warm square (nw x nw): paths between warm candidates never pass a
//     cold one (no outgoing edges), so it is the closure of W restricted to
//     them: repeated squaring on one thread-block cluster for up to
//     kClusterMaxWarm warm candidates, else the persistent blocked
//     Floyd-Warshall kernel below;
//   * the cold columns: p[i][c] = max(w[i][c], max_x min(p[i][x], w[x][c]))
//     over warm x, one (max, min) product with the closed warm square.
//
// When the caller's tally says the warm candidates are exactly the listed
// ones of a top-k profile (hint), every cold column is the same vector: for
// an unlisted c and a listed x, d[x][c] = cnt[x] (every ballot listing x puts
// it above c) and d[c][x] = 0, so w[x][c] = cnt[x] for all such c. The cold
// product then reduces to one column u[i] = max(w[i][c], max_x min(p[i][x],
// w[x][c])), which p, W's cold columns and beaten_by take from there.
//
// The persistent warm-square closure runs in rounds of B = 64 candidates; round r
//   1. closes the diagonal tile (r, r) by plain Floyd-Warshall,
//   2. updates the row and column panels: X = max(X, D (x) X) / max(X, X (x) D)
//      with D the closed diagonal tile,
//   3. updates every other tile: X(i, j) = max(X, W(i, r) (x) W(r, j)),
// where (x) is the (max, min) product. Widths only grow and every value
// written is the width of a real path, so the order of the updates inside a
// phase does not matter and the result is the exact closure. An update
// cannot change anything when min(max A, max B) <= min X over the tiles'
// entries, and is skipped; each tile's progress word carries its largest and
// smallest entry for that test. Updates left by it, of nb^3 (counted on the
// CPU, blocked Floyd-Warshall): 0.9% for Plackett-Luce Zipf(1.1) top-20 lists
// at m = 8192, 3.7% at m = 2048, 4.6% for top-200 lists at m = 2048, 2.1% for
// Mallows(0.98) full rankings and 92% for impartial culture at m = 1024. The
// closure went from 390 to 8.4 ms at m = 16384 (int32, top-20, 0.75% of the
// updates left, measured) and from 309 to 9.8 ms at m = 18407 (int16, top-200, 2.2%); it
// is now bound by the chain diagonal tile - panel - next diagonal tile of
// its 256 to 288 rounds (33 us each; 16 us where nothing else runs). Where
// every update is needed (uniform random d, int32) the tests and bounds cost
// 1% at m = 4096 (6.55 -> 6.62 ms without and with them), and larger squares
// gain from the shared operands of neighbouring tiles (m = 8192: 49.9 -> 48.5).
//
// All rounds run in ONE persistent cooperative launch: the CTAs take work
// items from a global queue in a fixed order in which the next round's
// diagonal and panel items come right after the current round's tiles in
// that row and column ("lookahead"), so they overlap the rest of the round.
// Each tile carries a progress word (rounds applied, bounds of its entries);
// an item, up to 32 tiles of one tile row or column, waits (bounded,
// clock-limited spin) until the tiles it reads have reached its round. Every wait is on an item earlier in the queue, which a
// resident CTA already holds, so the schedule cannot deadlock.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "internal.cuh"
#include "tiles.cuh"
#include "scan.cuh"

namespace schulze {
namespace {

using tiles::kB;        // block / tile size
using tiles::kThreads;  // threads per CTA
using tiles::BlockBarrier;
using tiles::Bounds;
using tiles::Ops;
using tiles::diag_closure_local;

// Progress word of a tile: rounds applied (12 bits), then the largest entry
// (rounded up) and the smallest (rounded down) as 26-bit values of
// 2^shift each.
constexpr int kBoundBits = 26;
constexpr uint32_t kBoundMax = (1u << kBoundBits) - 1u;

// The least shift at which the bound on the counts fits even rounded up: a
// clamped maximum could equal the rounded-down minimum of a tile that an
// update would still raise (bound 2^27 - 1: shift 2, not 1).
inline int word_shift(int64_t bound) {
  const int64_t top = bound < INT32_MAX ? bound : int64_t(INT32_MAX);
  int shift = 0;
  while ((top + (int64_t(1) << shift) - 1) >> shift > int64_t(kBoundMax)) ++shift;
  return shift;
}

__device__ __forceinline__ uint64_t make_word(uint32_t rounds, Bounds b, int shift) {
  // (the clamps act on entries above the bound alone, which are reported as SCHULZE_EDATA)
  const uint32_t mx = min((uint32_t(max(b.mx, 0)) + ((1u << shift) - 1u)) >> shift, kBoundMax);
  const uint32_t mn = min(uint32_t(max(b.mn, 0)) >> shift, kBoundMax);
  return (uint64_t(rounds) << (2 * kBoundBits)) | (uint64_t(mx) << kBoundBits) | mn;
}
__device__ __forceinline__ uint32_t word_rounds(uint64_t w) { return uint32_t(w >> (2 * kBoundBits)); }
__device__ __forceinline__ uint32_t word_max(uint64_t w) { return uint32_t(w >> kBoundBits) & kBoundMax; }
__device__ __forceinline__ uint32_t word_min(uint64_t w) { return uint32_t(w) & kBoundMax; }
__device__ __forceinline__ uint64_t word_at(uint64_t w, uint32_t rounds) {  // the same bounds, more rounds applied
  return (w & ((uint64_t(1) << (2 * kBoundBits)) - 1u)) | (uint64_t(rounds) << (2 * kBoundBits));
}

constexpr long long kSpinLimitCycles = 4000000000LL;  // ~2 s at 2 GHz, unless the context sets another

// ------------------------------------------------------------ relabel

// The weights in candidate order (w[i][j] as in pack_kernel, which permutes
// their rows and columns), kept in the output p until the widths replace them:
// rows of ldv entries of the closure's lane type, `vec` when each starts on a
// 16-byte boundary.
template <typename E>
struct Weights {
  E* v;
  int64_t ldv;
  int vec;
};
template <typename E>
Weights<E> weights_in(int32_t* p, int32_t m) {
  const size_t off = (16 - (reinterpret_cast<uintptr_t>(p) & 15u)) & 15u, room = size_t(m) * size_t(m) * 4;
  const size_t ldv = align_up(size_t(m) * sizeof(E), 16) / sizeof(E);
  if (off + size_t(m) * ldv * sizeof(E) <= room)
    return Weights<E>{reinterpret_cast<E*>(reinterpret_cast<char*>(p) + off), int64_t(ldv), 1};
  return Weights<E>{reinterpret_cast<E*>(p), int64_t(m), 0};
}

// With a valid hint the warm candidates are known. The weights are then
// gathered from d straight away (pack_kernel) where the warm square is small
// against the matrix: a gathered column costs a 32-byte sector per entry, so
// that above half of the candidates the two streaming passes read less.
__device__ __forceinline__ bool weigh_all(bool hv, int32_t nw, int32_t warm_max, int32_t m) {
  return !hv || (nw > warm_max && 2 * int64_t(nw) > m);
}

// rowflag[i] = the number of outgoing edges of candidate i (the j with
// d[i][j] > d[j][i]), and the weights in candidate order; also reports
// SCHULZE_EDATA for an entry outside [0, bound]. Each CTA takes 64 x 64 block
// pairs (A, B), A <= B: thread (r, c) holds d[A+r][B+c..c+3] and
// d[B+r][A+c..c+3] in registers (16-byte loads when rows are 16-byte
// aligned), both tiles go to shared memory, and each held entry is compared
// with its transposed partner from there. Bound by HBM (d read and the
// weights written once) as far as the instructions per entry allow: with a
// 64-bit test of every entry against the bound, the choice of weights made per
// entry and a shuffle sum per row it took 440 us at m = 16384 with 16-bit lanes
// and 479 with 32-bit ones, with one maximum per thread, kMargin and two rows
// per shuffle sum 300 and 343 (1.6 and 2.1 GB, 0.79 and 0.92 of HBM).
constexpr int kFlagT = 64;
template <typename E, bool kMargin>
__global__ void __launch_bounds__(256) weigh_kernel(const int32_t* __restrict__ d, int32_t m, int64_t bound,
                                                    int32_t* __restrict__ rowflag, int32_t* status,
                                                    const int32_t* __restrict__ warm,
                                                    const int32_t* __restrict__ hint_valid, int32_t warm_max, int vec4,
                                                    Weights<E> V) {
  pdl_enter_early();
  const bool hv = hint_valid && *hint_valid;
  if (!weigh_all(hv, hv ? *warm : 0, warm_max, m)) return;
  __shared__ int32_t t1[kFlagT][kFlagT + 1], t2[kFlagT][kFlagT + 1];  // t1 = d[A.., B..], t2 = d[B.., A..]
  const int32_t nbt = (m + kFlagT - 1) / kFlagT;
  const int64_t npairs = int64_t(nbt) * (nbt + 1) / 2;
  const int lane = threadIdx.x & 31;
  const int rq = threadIdx.x >> 4, c4 = (threadIdx.x & 15) * 4;  // rows rq + 16 q, columns c4 .. c4 + 3
  const bool vec = vec4 != 0;  // rows of d start on 16-byte boundaries
  int32_t a = 0;           // pairs (a, b), a <= b, numbered row by row
  int64_t rowstart = 0;    // number of the pair (a, a)
  uint32_t largest = 0;  // entry met, negative ones above every bound
  auto put = [&](int32_t i, int32_t j, const int32_t (&w)[4]) {  // weights of row i, columns j .. j + 3
    if (i >= m || j >= m) return;
    E* row = V.v + int64_t(i) * V.ldv + j;
    if (V.vec && sizeof(E) == 4) {
      *reinterpret_cast<int4*>(row) = make_int4(w[0], w[1], w[2], w[3]);
    } else if (V.vec) {  // (two 16-bit lanes per word; the row's padding takes zeros)
      *reinterpret_cast<uint2*>(row) = make_uint2((uint32_t(w[0]) & 0xFFFFu) | (uint32_t(w[1]) << 16),
                                                  (uint32_t(w[2]) & 0xFFFFu) | (uint32_t(w[3]) << 16));
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < m) row[e] = E(w[e]);
    }
  };
  for (int64_t t = blockIdx.x; t < npairs; t += gridDim.x) {
    while (t >= rowstart + (nbt - a)) rowstart += nbt - a, ++a;
    const int32_t A = a * kFlagT, B = (a + int32_t(t - rowstart)) * kFlagT;
    int32_t x1[4][4], x2[4][4];
    auto load = [&](int32_t R, int32_t Cc, int32_t (&x)[4][4]) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int32_t i = R + rq + 16 * q, j = Cc + c4;
        if (vec) {
          int4 v = make_int4(0, 0, 0, 0);
          if (i < m && j < m) v = __ldcs(reinterpret_cast<const int4*>(d + int64_t(i) * m + j));
          x[q][0] = v.x, x[q][1] = v.y, x[q][2] = v.z, x[q][3] = v.w;
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) x[q][e] = (i < m && j + e < m) ? d[int64_t(i) * m + j + e] : 0;
        }
        largest = max(largest, max(max(uint32_t(x[q][0]), uint32_t(x[q][1])), max(uint32_t(x[q][2]), uint32_t(x[q][3]))));
      }
    };
    load(A, B, x1);
    if (A != B) load(B, A, x2);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        t1[rq + 16 * q][c4 + e] = x1[q][e];
        if (A != B) t2[rq + 16 * q][c4 + e] = x2[q][e];
      }
    __syncthreads();
    // side 0: row A + r, columns B + c: edge when t1[r][c] > (t2 or t1)[c][r]
    // side 1: row B + r, columns A + c: edge when t2[r][c] > t1[c][r]
    const int32_t(*T)[kFlagT + 1] = A == B ? t1 : t2;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t e = 0;  // edges of rows 2 h and 2 h + 1 of side 0, then of side 1 (64 at most each), a byte each
#pragma unroll
      for (int q = 2 * h; q < 2 * h + 2; ++q) {
        const int r = rq + 16 * q;
        const uint32_t one = q & 1 ? 0x100u : 1u;
        int32_t w[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {  // (on the diagonal both sides are the same entry: no edge)
          const int32_t u = T[c4 + x][r];
          const bool edge = x1[q][x] > u;
          e += edge ? one : 0u;
          w[x] = edge ? x1[q][x] - (kMargin ? u : 0) : 0;
        }
        put(A + r, B + c4, w);
        if (A != B) {
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const int32_t u = t1[c4 + x][r];
            const bool edge = x2[q][x] > u;
            e += edge ? one << 16 : 0u;
            w[x] = edge ? x2[q][x] - (kMargin ? u : 0) : 0;
          }
          put(B + r, A + c4, w);
        }
      }
      // padding entries are 0 on both sides, so they never count
#pragma unroll
      for (int o = 8; o; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
      const int r = rq + 32 * h + (lane & 1) * 16, f = int(e >> (lane & 1) * 8);
      if ((lane & 15) < 2) {
        if (f & 0xFF) atomicAdd(&rowflag[A + r], f & 0xFF);
        if ((f >> 16) & 0xFF) atomicAdd(&rowflag[B + r], (f >> 16) & 0xFF);
      }
    }
    __syncthreads();
  }
  if (largest > uint32_t(min(bound, int64_t(INT32_MAX)))) set_status(status, SCHULZE_EDATA);
}

// perm[new] = old, inv[old] = new: candidates with edges first, strongest
// first, then the others in id order. Strength is the number of outgoing
// edges (weigh_kernel), or, when the tally set *hint_valid, the number of
// ballots that list the candidate (hint). It is sorted by counting over
// kStrengths classes (equal sizes for edge counts, relative steps of 1/128
// for ballots; any order inside a class): the closure needs like candidates
// near each other, not an exact order. The tally has written a warm-first
// relabeling already when its hint is valid; it is kept where the cluster
// closure takes the whole warm square (warm_max), whose cost does not depend
// on the order, and without a hint such a set stays in id order too.
constexpr int kStrengths = 4096;

__device__ __forceinline__ int strength_class(uint32_t x, bool ballots, int32_t m) {
  if (ballots) {  // x >= 1: exponent and the seven bits after the leading one
    const int lz = __clz(x);
    return kStrengths - 1 - ((31 - lz) * 128 + int((x << lz >> 24) & 127u));
  }
  return kStrengths - 1 - int(uint64_t(x) * kStrengths / uint64_t(m));  // x < m
}

__global__ void __launch_bounds__(1024) relabel_kernel(const int32_t* __restrict__ rowflag, int32_t m,
                                                       int32_t* __restrict__ perm, int32_t* __restrict__ inv,
                                                       int32_t* __restrict__ warm_out,
                                                       const int32_t* __restrict__ hint,
                                                       const int32_t* __restrict__ hint_valid, int32_t warm_max) {
  pdl_enter_early();
  __shared__ uint32_t part[33];
  __shared__ uint32_t cls[kStrengths];
  extern __shared__ uint32_t relabel_smem[];  // m words when m <= kScanSmem
  const bool hv = hint_valid && *hint_valid;
  if (hv && *warm_out <= warm_max) return;
  const int32_t* strength = hv ? hint : rowflag;
  // rank[c] = 1 for warm c, scanned into the warm rank (in shared memory, or
  // in place in inv for long candidate lists)
  uint32_t* rank = m <= kScanSmem ? relabel_smem : reinterpret_cast<uint32_t*>(inv);
  for (int32_t c = threadIdx.x; c < m; c += blockDim.x) rank[c] = strength[c] ? 1u : 0u;
  __syncthreads();
  const int32_t warm = int32_t(block_exclusive_scan(rank, m, part));
  const bool sorted = warm > warm_max;
  if (sorted) {
    for (int t = threadIdx.x; t < kStrengths; t += blockDim.x) cls[t] = 0u;
    __syncthreads();
    for (int32_t c = threadIdx.x; c < m; c += blockDim.x) {
      const int32_t x = strength[c];
      if (x) atomicAdd(&cls[strength_class(uint32_t(x), hv, m)], 1u);
    }
    __syncthreads();
    block_exclusive_scan(cls, kStrengths, part);
  }
  if (threadIdx.x == 0) *warm_out = warm;
  for (int32_t c = threadIdx.x; c < m; c += blockDim.x) {
    const int32_t x = strength[c];
    const int32_t nw = !x ? warm + (c - int32_t(rank[c]))  // rank[c] warm candidates before c
                       : !sorted ? int32_t(rank[c])
                                 : int32_t(atomicAdd(&cls[strength_class(uint32_t(x), hv, m)], 1u));
    perm[nw] = c;
    inv[c] = nw;
  }
}

// W[a][b] = w[perm[a]][perm[b]] for the warm rows a < 64 * nbr (0 outside
// m x m, on the diagonal and where d does not beat its transpose; w is d, or
// the margin d - d^T with `margin`), with the bounds of the 64 x 64 tiles in
// tmax and tmin (tmin holds INT32_MAX - min, so that both start at zero): the
// largest entry, and the smallest one among the warm rows and the existing
// columns, off the diagonal. With uniform cold columns only the square
// (b < 64 nbr) is written, and ucol[a] receives the cold columns' common
// value for row a.
//
// Two forms. After weigh_kernel, a CTA copies row perm[a] of the weights to
// shared memory (when it fits, `rowbuf` bytes) and gathers its columns from
// there, eight per thread: both passes over the matrix stay coalesced
// whatever the order (gathering d's columns in strength order took 7.1 ms at
// m = 16384, int32, a 32-byte sector per entry; weigh_kernel and this form
// take 0.36 + 0.65 ms). Else (few warm
// candidates) with x = perm[a] the threads read d[x][perm b] (along row x) and
// d[perm b][x] (down column x); a candidate y without edges is one no ballot
// lists, so d[y][x] = 0 and that read is skipped. `chunk` rows (of one tile
// row) per CTA pass.
template <typename E>
__global__ void __launch_bounds__(512) pack_kernel(const int32_t* __restrict__ d, int32_t m, int32_t mp,
                                                   const int32_t* __restrict__ perm, const int32_t* __restrict__ warm,
                                                   E* __restrict__ W, int32_t* __restrict__ tmax,
                                                   int32_t* __restrict__ tmin, int32_t nb,
                                                   const int32_t* __restrict__ hint,
                                                   const int32_t* __restrict__ hint_valid, int32_t* __restrict__ ucol,
                                                   int margin, int32_t warm_max, Weights<E> V, uint32_t rowbuf,
                                                   int32_t chunk) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char pack_smem[];
  const bool hv = hint_valid && *hint_valid;
  const int32_t nw = *warm;
  const int32_t rows = (nw + kB - 1) / kB * kB;  // W rows to write
  const bool uc = hv && rows < m;                    // uniform cold columns beyond the square
  const int32_t bend = uc ? rows : mp;
  const int lane = threadIdx.x & 31;
  if (weigh_all(hv, nw, warm_max, m)) {
    // few warm candidates: spread them (m = 8192, 144 warm, no hint: 48 -> 11 us)
    while (chunk > 1 && rows < chunk * int32_t(gridDim.x)) chunk >>= 1;
    E* srow = reinterpret_cast<E*>(pack_smem);
    int32_t* cmax = reinterpret_cast<int32_t*>(pack_smem + rowbuf);  // this chunk's bounds per tile column
    int32_t* cmin = cmax + nb;
    for (int t = threadIdx.x; t < 2 * nb; t += blockDim.x) cmax[t] = 0;
    for (int32_t a0 = int32_t(blockIdx.x) * chunk; a0 < rows; a0 += int32_t(gridDim.x) * chunk) {
      for (int32_t a = a0; a < a0 + chunk; ++a) {
        E* wrow = W + int64_t(a) * mp;
        __syncthreads();  // the row before is read
        if (a >= nw) {    // rows without edges up to a whole tile
          for (int32_t b = 8 * threadIdx.x; b < bend; b += 8 * blockDim.x) {
#pragma unroll
            for (int e = 0; e < int(sizeof(E)) / 2; ++e) reinterpret_cast<uint4*>(wrow + b)[e] = make_uint4(0, 0, 0, 0);
          }
          continue;
        }
        const int32_t x = perm[a];
        if (uc && threadIdx.x == 0) ucol[a] = max(d[int64_t(x) * m + perm[rows]], 0);
        const E* vrow = V.v + int64_t(x) * V.ldv;
        if (rowbuf) {
          if (V.vec) {
            const int32_t n16 = int32_t((size_t(m) * sizeof(E) + 15) / 16);
            for (int32_t t0 = threadIdx.x; t0 < n16; t0 += 4 * blockDim.x) {
              uint4 v[4];
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (t0 + q * int32_t(blockDim.x) < n16) v[q] = __ldcs(reinterpret_cast<const uint4*>(vrow) + t0 + q * blockDim.x);
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (t0 + q * int32_t(blockDim.x) < n16) reinterpret_cast<uint4*>(srow)[t0 + q * blockDim.x] = v[q];
            }
          } else {
            for (int32_t t = threadIdx.x; t < m; t += blockDim.x) srow[t] = vrow[t];
          }
          __syncthreads();
          vrow = srow;
        }
        for (int32_t b = 8 * threadIdx.x; b < bend; b += 8 * blockDim.x) {
          int32_t w[8], mx = 0, mn = INT32_MAX;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            w[e] = b + e < m ? int32_t(vrow[perm[b + e]]) : 0;
            mx = max(mx, w[e]);
            if (b + e < m && b + e != a) mn = min(mn, w[e]);
          }
          if (sizeof(E) == 2) {
            uint32_t u[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) u[e] = (uint32_t(w[2 * e]) & 0xFFFFu) | (uint32_t(w[2 * e + 1]) << 16);
            *reinterpret_cast<uint4*>(wrow + b) = make_uint4(u[0], u[1], u[2], u[3]);
          } else {
            reinterpret_cast<int4*>(wrow + b)[0] = make_int4(w[0], w[1], w[2], w[3]);
            reinterpret_cast<int4*>(wrow + b)[1] = make_int4(w[4], w[5], w[6], w[7]);
          }
          if (mx > 0) atomicMax(&cmax[b / kB], mx);
          if (mn < INT32_MAX) atomicMax(&cmin[b / kB], INT32_MAX - max(mn, 0));
        }
      }
      __syncthreads();
      for (int t = threadIdx.x; t < bend / kB; t += blockDim.x) {
        if (cmax[t]) atomicMax(&tmax[(a0 / kB) * nb + t], cmax[t]), cmax[t] = 0;
        if (cmin[t]) atomicMax(&tmin[(a0 / kB) * nb + t], cmin[t]), cmin[t] = 0;
      }
    }
    return;
  }
  constexpr int kU = 8;  // columns per thread and pass, their loads issued together
  for (int32_t a = blockIdx.x; a < rows; a += gridDim.x) {
    E* wrow = W + int64_t(a) * mp;
    const int32_t x = a < m ? perm[a] : -1;
    const int32_t* drow = x >= 0 ? d + int64_t(x) * m : nullptr;
    if (uc && threadIdx.x == 0) ucol[a] = (x >= 0 && a < nw) ? max(drow[perm[rows]], 0) : 0;
    for (int32_t b0 = 0; b0 < bend; b0 += kU * blockDim.x) {
      int32_t y[kU], v[kU], u[kU];
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        const int32_t b = b0 + q * blockDim.x + threadIdx.x;
        y[q] = (x >= 0 && b < m && b < bend && b != a) ? perm[b] : -1;
      }
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        v[q] = y[q] >= 0 ? drow[y[q]] : 0;
        u[q] = (y[q] >= 0 && !(hv && !hint[y[q]])) ? d[int64_t(y[q]) * m + x] : 0;
      }
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        const int32_t b = b0 + q * blockDim.x + threadIdx.x;
        const int32_t out = v[q] > u[q] ? (margin ? v[q] - u[q] : v[q]) : 0;
        if (b < bend) wrow[b] = E(out);
        const int32_t mx = __reduce_max_sync(0xFFFFFFFFu, out);
        const int32_t mn = __reduce_min_sync(0xFFFFFFFFu, a < nw && b < m && b != a ? out : INT32_MAX);
        if (lane == 0 && b < bend) {
          const int32_t t = (a / kB) * nb + b / kB;
          if (mx > 0) atomicMax(&tmax[t], mx);
          if (mn < INT32_MAX) atomicMax(&tmin[t], INT32_MAX - max(mn, 0));
        }
      }
    }
  }
}

// p[x][y] = W[inv[x]][inv[y]] for warm x and y != x; every other entry 0
// (cold rows are written as zeros without reading W). A warm row of W is
// copied to shared memory (when it fits, `rowbuf` bytes) and gathered from
// there, so that W and p are both streamed whatever the order; bound by HBM
// (m = 16384, int32: 0.61 ms for 2.1 GB, against 1.47 gathering from global
// memory in strength order; m = 18407, int16: 0.64 against 2.05 ms).
// With uniform cold columns (uc) every column outside the square is ucold.
template <typename E>
__global__ void __launch_bounds__(512) widen_kernel(const E* __restrict__ W, int32_t mp, int32_t m,
                                                    const int32_t* __restrict__ inv,
                                                    const int32_t* __restrict__ perm,
                                                    const int32_t* __restrict__ warm, int32_t* __restrict__ p,
                                                    const int32_t* __restrict__ hint_valid,
                                                    const int32_t* __restrict__ ucold, int vec4, uint32_t rowbuf) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char widen_smem[];
  const int32_t nw = *warm;
  const int32_t rows = (nw + kB - 1) / kB * kB;
  const bool uc = hint_valid && *hint_valid && rows < m;  // cold columns beyond the square: ucold[ix]
  // kR rows per pass: their relabeled indices are loaded together (lane r of
  // each warp holds row r's) instead of one dependent load per row
  constexpr int kR = 8;
  const int lane = threadIdx.x & 31;
  for (int32_t xb = blockIdx.x; xb < m; xb += kR * gridDim.x) {
    const int32_t xl = xb + lane * int32_t(gridDim.x);
    const int32_t ixl = (lane < kR && xl < m) ? inv[xl] : 0;
    for (int r = 0; r < kR; ++r) {
      const int32_t x = xb + r * int32_t(gridDim.x);
      if (x >= m) break;
      const int32_t ix = __shfl_sync(0xFFFFFFFFu, ixl, r);
      int32_t* prow = p + int64_t(x) * m;
      const E* wrow = W + int64_t(ix) * mp;
      // a cold row is zero; with uniform cold columns and a small square a
      // warm row is ucold[ix] outside the square, whose columns (relabeled
      // b < rows, candidate perm[b]) come from W after the fill
      if (ix >= nw || (uc && 4 * rows < m)) {
        const int32_t fill = ix >= nw ? 0 : ucold[ix];
        if (vec4) {
          for (int32_t y = 4 * threadIdx.x; y < m; y += 4 * blockDim.x)
            *reinterpret_cast<int4*>(prow + y) = make_int4(fill, fill, fill, fill);
        } else {
          for (int32_t y = threadIdx.x; y < m; y += blockDim.x) prow[y] = fill;
        }
        if (ix >= nw) continue;
        __syncthreads();  // the square's columns after the fill (the branch is the same in the whole CTA)
        for (int32_t b = threadIdx.x; b < rows; b += blockDim.x) prow[perm[b]] = b == ix ? 0 : int32_t(wrow[b]);
        continue;
      }
      const int32_t lim = uc ? rows : mp;  // columns of W to read
      const int32_t uv = uc ? ucold[ix] : 0;
      if (rowbuf) {
        __syncthreads();  // the row before is read
        E* srow = reinterpret_cast<E*>(widen_smem);
        const int32_t n16 = lim * int32_t(sizeof(E)) / 16;  // (whole tiles)
        for (int32_t t0 = threadIdx.x; t0 < n16; t0 += 4 * blockDim.x) {
          uint4 v[4];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (t0 + q * int32_t(blockDim.x) < n16) v[q] = __ldcs(reinterpret_cast<const uint4*>(wrow) + t0 + q * blockDim.x);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (t0 + q * int32_t(blockDim.x) < n16) reinterpret_cast<uint4*>(srow)[t0 + q * blockDim.x] = v[q];
        }
        __syncthreads();
        wrow = srow;
      }
      constexpr int kU = 8;
      for (int32_t y0 = threadIdx.x; y0 < m; y0 += kU * blockDim.x) {
        int32_t iy[kU], v[kU];
#pragma unroll
        for (int q = 0; q < kU; ++q) iy[q] = y0 + q * int32_t(blockDim.x) < m ? inv[y0 + q * blockDim.x] : 0;
#pragma unroll
        for (int q = 0; q < kU; ++q) v[q] = iy[q] < lim ? int32_t(wrow[iy[q]]) : uv;
#pragma unroll
        for (int q = 0; q < kU; ++q) {
          const int32_t y = y0 + q * int32_t(blockDim.x);
          if (y < m) __stcs(prow + y, y == x ? 0 : v[q]);
        }
      }
    }
  }
}

// ----------------------------------------------------- work queue

enum ItemKind : int32_t { kDiag = 0, kPanel = 1, kTile = 2, kStop = 3 };

// A work item: cnt tiles in round r, with the running index v0 + t * stride
// for tile t. The index runs along tile row or column fix, or (kGrid) over
// the n x n tiles of R(r) row by row; tile indices are counted without the
// `skip` indices r, r + 1, ...
constexpr int kItemTiles = 32;  // one per lane
enum ItemShape : int32_t { kRow = 0, kColumn = 1, kGrid = 2 };
struct Item {
  int32_t kind, r, shape, fix, v0, stride, cnt, skip, n;
  __device__ __forceinline__ void tile(int32_t t, int32_t& i, int32_t& j) const {
    int32_t x = v0 + t * stride, y = fix;
    if (shape == kGrid) y = x / n, x -= y * n, y = y < r ? y : y + skip;
    x = x < r ? x : x + skip;
    i = shape == kColumn ? x : y, j = shape == kColumn ? y : x;
  }
};

// The candidates with outgoing edges occupy the first nbr tile rows after
// relabeling; the other rows of W are zero and stay zero, and a round over a
// block of them cannot change anything (min(x, 0) = 0). So rounds run over
// r < nbr on the nbr x nbr tiles of the warm square; cold_product_kernel does
// the cold columns.
//
// Queue order, stage by stage:
//   stage 0:             D(0) P(0) D(1) L(0)
//   stage s (1..nbr-2):  P(s) X(s-1) D(s+1) L(s) R(s-1)
//   stage nbr-1:         P(s) R(s-1)
//   stage nbr:           R(nbr-1)
// D(r): the diagonal tile: its round r-1 update, then its closure; P(r): the
// panel tiles (r, r+1) and (r+1, r) that D(r+1) waits for, then the rest of
// row panel r and of column panel r; L(r): the round-r tiles of tile row and
// column r+1, which the next round's panels are made of; X(r): those of tile
// row and column r+2, which L(r+1) is made of; R(r): the other round-r tiles.
// So the chain from one diagonal tile to the next (D, P, D, ...) never waits
// for R, and D(r+1) runs beside R(r-1). P, L and X come tile by tile, which
// keeps the chain of the panels short, R in items of at most gr tiles: about
// two items per CTA and round. The tests of 32
// tiles, a lane each, cost one round trip to the progress words instead of 32
// (a skipped tile by itself would take its CTA about a microsecond); 64 left
// the items with too much work (m = 18407 top-200: 12.9 ms against 9.7). The
// tiles of an item are spread evenly over their range: those that need an
// update lie next to each other (m = 16384 top-20: 480 of 65536 in a round),
// and items of neighbours left some CTAs with most of them (the closure took
// 28.5 ms, 10.8 ms spread).
// Where most tiles need their update (run) none of that holds: the tiles of an
// item are then neighbours along a tile row, which share their operand (i, r),
// and there are about eight items per CTA and round (fewer tiles, and the tests
// cost too much; more, and a round ends with CTAs waiting for its last items),
// at least pairs of tiles from four tiles per CTA on. Uniform random d, int32,
// spread and one tile per item up to m = 8192 against this: m = 4096 6.69 -> 6.62
// ms, m = 5000 12.42 -> 11.99, m = 8192 51.7 -> 48.5, m = 12288 167.5 -> 159.6;
// int16, m = 8192: 27.7 -> 25.6.
struct Shape {
  int32_t nbr, gr;
  bool run;
  int32_t P, L;         // items of P(r), L(r), r < nbr - 1
  int32_t X, R;         // items of X(r), R(r), r < nbr - 2
  int32_t P_last, R_pen, R_last;  // P(nbr - 1), R(nbr - 2), R(nbr - 1)
  uint32_t first, mid, total;     // items of stage 0, of a stage 1 .. nbr - 2, of the queue
};

__device__ Shape make_shape(int32_t nbr, int32_t grid, bool dense) {  // nbr >= 3
  Shape sh;
  sh.nbr = nbr, sh.run = dense;
  const int32_t per = nbr * nbr / grid;  // tiles per CTA and round
  sh.gr = min(kItemTiles, !dense ? max(1, per / 2) : per >= 4 ? max(2, per / 8) : 1);
  const int32_t q = nbr - 2;  // tile indices without r and r + 1
  sh.P = 2 + 2 * q, sh.L = 2 * q, sh.P_last = 2 * (q + 1);
  sh.X = q + (q - 1), sh.R = ((q - 1) * (q - 1) + sh.gr - 1) / sh.gr;
  sh.R_pen = (q * q + sh.gr - 1) / sh.gr, sh.R_last = ((q + 1) * (q + 1) + sh.gr - 1) / sh.gr;
  sh.first = 2 + sh.P + sh.L, sh.mid = 1 + sh.P + sh.X + sh.L + sh.R;
  sh.total = sh.first + uint32_t(q) * sh.mid + uint32_t(sh.P_last + sh.R_pen + sh.R_last);
  return sh;
}

// item t of the queue, t < sh.total
__device__ Item decode_item(uint32_t t, const Shape& sh) {
  const int32_t nbr = sh.nbr, q = nbr - 2;
  int32_t s = 0;
  if (t >= sh.first) {
    t -= sh.first;
    if (t < uint32_t(q) * sh.mid) {
      s = 1 + int32_t(t / sh.mid);
      t -= uint32_t(s - 1) * sh.mid;
    } else {
      t -= uint32_t(q) * sh.mid;
      s = nbr - 1;
      const uint32_t z = sh.P_last + sh.R_pen;
      if (t >= z) t -= z, s = nbr;
    }
  }
  auto one = [](int32_t kind, int32_t r, int32_t i, int32_t j) { return Item{kind, r, kRow, i, j, 0, 1, 0, 0}; };
  // item a of a tile row's or column's; item a of the `items` of a grid
  auto side = [](int32_t kind, int32_t r, int32_t shape, int32_t fix, int32_t a, int32_t skip) {
    return Item{kind, r, shape, fix, a, 0, 1, skip, 0};
  };
  auto grid = [&](int32_t r, int32_t a, int32_t items, int32_t n, int32_t skip) {
    return Item{kTile, r, kGrid, 0, sh.run ? a * sh.gr : a, sh.run ? 1 : items, sh.gr, skip, n};
  };
  int32_t a = int32_t(t);
  if (s == nbr) return grid(nbr - 1, a, sh.R_last, q + 1, 1);
  if (s == nbr - 1) {
    if (a < sh.P_last)
      return side(kPanel, s, a <= q ? kRow : kColumn, s, a <= q ? a : a - (q + 1), 1);
    return grid(s - 1, a - sh.P_last, sh.R_pen, q, 2);
  }
  if (s == 0) {
    if (a == 0) return one(kDiag, 0, 0, 0);
    a -= 1;
  }
  if (a < 2) return a == 0 ? one(kPanel, s, s, s + 1) : one(kPanel, s, s + 1, s);
  if (a < sh.P) {
    a -= 2;
    return side(kPanel, s, a < q ? kRow : kColumn, s, a < q ? a : a - q, 2);
  }
  a -= sh.P;
  if (s >= 1) {
    if (a < q) return side(kTile, s - 1, kRow, s + 1, a, 2);
    if (a < sh.X) return side(kTile, s - 1, kColumn, s + 1, a - q, 3);
    a -= sh.X;
  }
  if (a == 0) return one(kDiag, s + 1, s + 1, s + 1);
  a -= 1;
  if (a < sh.L) return side(kTile, s, a < q ? kRow : kColumn, s + 1, a < q ? a : a - q, 2);
  return grid(s - 1, a - sh.L, sh.R, q - 1, 3);
}

struct Sync {
  unsigned long long* prog;      // [nb * nb] progress words
  const int32_t* tmax;           // [nb * nb] bounds of the packed tiles (pack_kernel)
  const int32_t* tmin;
  uint32_t* head;                // queue head
  uint32_t* abort_flag;          // set when a wait times out
  int32_t* status;
  const int32_t* warm;           // candidates with outgoing edges
  unsigned long long* counters;  // [0] tile updates done, [1] diagonal closures done, [2] items
  long long spin_limit;          // clock cycles a wait may take before it gives up
  int32_t shift;                 // progress word bounds are in units of 2^shift
};

// Progress words are read and written relaxed, with one fence between the
// reads an item waits for and its work, and one between the work and its word
// (an acquire per read would make the three reads of a test wait for one
// another).
__device__ __forceinline__ uint64_t load_word(const unsigned long long* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// (__threadfence() would be the stronger, slower fence.sc)
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void store_word(unsigned long long* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Warm squares up to this size are closed by closure_cluster_kernel (the
// square must fit one CTA's shared memory), larger ones by the persistent
// kernel.
template <typename E>
constexpr int32_t kClusterMaxWarm = sizeof(E) == 2 ? 256 : 192;

// CTAs per SM: five for int32 lanes (at most 96 registers a thread), which
// measured fastest against four and six; six for packed int16 lanes (80
// registers; seven spill, uniform random d at m = 1000: 0.506 against 0.474
// ms for the whole call, m = 8192: 29.15 against 29.41 ms)
#define SCHULZE_PERSIST_BOUNDS __launch_bounds__(kThreads, sizeof(E) == 2 ? 6 : 5)

// Warp 1 runs the schedule: it claims the CTA's next queue slot while the CTA
// works on the current item, and between items its lanes wait for the words
// the new item's tiles depend on (own tile: the rounds before; panel: the
// closed diagonal; tile: both panels; diagonal: both panels of the round
// before) and test their bounds: a tile that cannot change is passed on to
// the next round at once, the others are computed one after another by the
// CTA and published by thread 0 as they are done (the last one while warp 1 is
// at the next item already). The schedule stays deadlock-free: every wait is
// on an item earlier in the queue, and a CTA holds at most one claimed,
// unstarted item, later in the queue than its current one, so the earliest
// unfinished item is always being worked on.
struct Slot {  // an item and its tiles to compute; diagonal: whether its update of the round before is needed
  Item it;
  uint32_t mask, update;
};

// warp 1: the item of queue slot t into *s (kStop at the end of the queue or
// after a failed wait); out of line, as the tile update needs the registers
__device__ __noinline__ void next_item(const Sync& sy, uint32_t t, const Shape& sh, int32_t nb, Slot* s) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    if (t >= sh.total || *reinterpret_cast<volatile uint32_t*>(sy.abort_flag)) s->it = Item{kStop, 0, kRow, 0, 0, 0, 0, 0, 0};
    else s->it = decode_item(t, sh);
  }
  __syncwarp();
  const Item it = s->it;
  const uint32_t r = uint32_t(it.r);
  const bool diag = it.kind == kDiag;
  // rounds the own word and the operands' words need to have; a diagonal
  // tile's own update is that of round r - 1
  const uint32_t n0 = diag && r ? r - 1 : r, nd = diag ? r : r + 1;
  const int32_t rr = diag ? it.r - 1 : it.r;  // the round whose operands are read
  const bool two = it.kind == kTile || (diag && r);  // operands (i, rr) and (rr, j)
  bool ok = true, need = false, update = false;
  if (lane < it.cnt && (it.shape != kGrid || it.v0 + lane * it.stride < it.n * it.n)) {
    int32_t i, j;
    it.tile(lane, i, j);
    const int32_t own = i * nb + j;
    const int32_t da = it.kind == kPanel ? it.r * nb + it.r : i * nb + rr, db = rr * nb + j;
    constexpr uint64_t kThere = ~uint64_t(0);  // (no word to wait for)
    uint64_t w0 = n0 ? load_word(sy.prog + own) : kThere;
    uint64_t w1 = two || it.kind == kPanel ? load_word(sy.prog + da) : kThere;
    uint64_t w2 = two ? load_word(sy.prog + db) : kThere;
    const long long t0 = clock64();
    for (;;) {
      const bool m0 = word_rounds(w0) < n0, m1 = word_rounds(w1) < nd, m2 = word_rounds(w2) < nd;
      if (!(m0 || m1 || m2)) break;
      if (*reinterpret_cast<volatile uint32_t*>(sy.abort_flag)) ok = false;
      if (ok && clock64() - t0 > sy.spin_limit) {
        set_status(sy.status, SCHULZE_ETIMEOUT);
        atomicExch(sy.abort_flag, 1u);
        ok = false;
      }
      if (!ok) break;
      __nanosleep(32);
      if (m0) w0 = load_word(sy.prog + own);
      if (m1) w1 = load_word(sy.prog + da);
      if (m2) w2 = load_word(sy.prog + db);
    }
    fence_gpu();
    if (n0 == 0) w0 = make_word(0, Bounds{sy.tmax[own], INT32_MAX - sy.tmin[own]}, sy.shift);
    // what the update can offer at most, against the tile's smallest entry
    const uint32_t offer = min(word_max(w1), two ? word_max(w2) : word_max(w0));
    need = offer > word_min(w0);
    if (diag) {
      update = two && need;
      need = update || word_max(w0) > 0;  // a zero tile is closed
    }
    if (ok && !need) store_word(sy.prog + own, word_at(w0, r + 1));
  }
  const uint32_t mask = __ballot_sync(0xFFFFFFFFu, need), fail = __ballot_sync(0xFFFFFFFFu, !ok);
  if (lane == 0) {
    s->mask = mask, s->update = update ? 1u : 0u;
    if (fail) s->it.kind = kStop;
  }
}

// Whether at least three quarters of the tile updates look needed: 128
// triples of tiles, tested on the packed bounds (every CTA samples the same
// ones).
__device__ __forceinline__ bool sample_dense(const Sync& sy, int32_t nbr, int32_t nb) {
  uint32_t h = (threadIdx.x + 1u) * 2654435761u;
  auto draw = [&]() {
    h ^= h >> 15, h *= 2246822519u, h ^= h >> 13;
    return int32_t(h % uint32_t(nbr));
  };
  const int32_t i = draw(), k = draw(), j = draw();
  const bool need = min(sy.tmax[i * nb + k], sy.tmax[k * nb + j]) > INT32_MAX - sy.tmin[i * nb + j];
  return __syncthreads_count(need) >= kThreads * 3 / 4;
}

template <typename E>
__global__ void SCHULZE_PERSIST_BOUNDS closure_persistent_kernel(E* W, int32_t ld, int32_t m, int32_t nb,
                                                                 const __grid_constant__ Sync sy) {
  pdl_enter_early();
  __shared__ __align__(16) typename Ops<E>::Smem sm;
  __shared__ __align__(16) int32_t rowbuf[2][kB];
  __shared__ Shape s_shape;
  // two slots: warp 1 writes the next one while the others read the current
  __shared__ Slot s_slot[2];
  __shared__ uint32_t s_done[3];  // tile updates, diagonal closures, items
  __shared__ Bounds s_bd[2][kThreads / 32];
  const int32_t nw = *sy.warm;
  if (nw <= kClusterMaxWarm<E>) return;  // closure_cluster_kernel's case
  const int32_t nbr = (nw + kB - 1) / kB;  // nb is the progress words' row stride
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool dense = sample_dense(sy, nbr, nb);
  if (tid < 3) s_done[tid] = 0u;
  if (tid == 32) s_shape = make_shape(nbr, int32_t(gridDim.x), dense);  // (warp 1 alone reads it)
  __syncwarp();
  uint32_t next = 0;  // warp 1, lane 0: the claimed queue slot
  if (tid == 32) next = atomicAdd(sy.head, 1u);
  for (int buf = 0, par = 0;; buf ^= 1) {
    if (wid == 1) next_item(sy, next, s_shape, nb, &s_slot[buf]);
    __syncthreads();
    const Slot& sl = s_slot[buf];
    const int32_t kind = sl.it.kind, r = sl.it.r;
    if (kind == kStop) break;
    if (tid == 32) next = atomicAdd(sy.head, 1u), ++s_done[2];  // in flight during this item
    int32_t cur_a = -1, cur_b = -1;  // staged operand tiles: (cur_a, r) and (r, cur_b)
    for (uint32_t mask = sl.mask; mask; mask &= mask - 1) {
      int32_t i, j;
      sl.it.tile(__ffs(int(mask)) - 1, i, j);
      Bounds bd;
      const int32_t vr = nw - i * kB, vc = m - j * kB;  // candidates with edges / candidates from the tile's corner on
      E* Cg = W + int64_t(i) * kB * ld + int64_t(j) * kB;
      if (kind == kDiag) {
        if (sl.update) {  // its update of the round before
          Ops<E>::load_a(Cg - kB, ld, sm, tid);
          Ops<E>::load_b(Cg - int64_t(kB) * ld, ld, sm, tid);
          Ops<E>::template multiply<false>(Cg, ld, sm, tid, BlockBarrier{}, bd);
          __syncthreads();
        }
        diag_closure_local<E>(W, ld, r, vr, vc, rowbuf, tid, BlockBarrier{}, bd);
      } else {
        // the tiles of a panel side share an operand
        if (cur_a != i) Ops<E>::load_a(W + int64_t(i) * kB * ld + int64_t(r) * kB, ld, sm, tid);
        if (cur_b != j) Ops<E>::load_b(W + int64_t(r) * kB * ld + int64_t(j) * kB, ld, sm, tid);
        cur_a = i, cur_b = j;
          Ops<E>::template multiply<true>(Cg, ld, sm, tid, BlockBarrier{}, bd, i == j || vr < kB || vc < kB, i == j,
                                          vr, vc);
      }
      const int32_t mx = __reduce_max_sync(0xFFFFFFFFu, bd.mx), mn = __reduce_min_sync(0xFFFFFFFFu, bd.mn);
      if (lane == 0) s_bd[par][wid] = Bounds{mx, mn};
      __syncthreads();  // every store of the tile and its bounds done, operands free
      if (tid == 0) {
        Bounds b = s_bd[par][0];
#pragma unroll
        for (int w = 1; w < kThreads / 32; ++w) b.mx = max(b.mx, s_bd[par][w].mx), b.mn = min(b.mn, s_bd[par][w].mn);
        fence_gpu();
        store_word(sy.prog + (i * nb + j), make_word(r + 1, b, sy.shift));
        ++s_done[kind == kDiag ? 1 : 0];
      }
      par ^= 1;
    }
  }
  __syncthreads();
  if (tid < 3) atomicAdd(&sy.counters[tid], (unsigned long long)s_done[tid]);
}

// Warm squares of at most kClusterMaxWarm candidates: the closure by
// repeated (max, min) squaring, in place, on a cluster of kClusterCtas CTAs
// (one per SM). Every CTA holds a copy of the square S (n = nw rounded up to
// 64, row-major) in shared memory; CTA q owns the warm rows q, q + 8, ... A
// sweep sets, for every owned row i and column j,
//   S[i][j] = max(S[i][j], max_{k < nw} min(S[i][k], S[k][j])),
// reading whatever the copy holds: widths only grow and every value is the
// width of a real path, so a mix of older and newer entries is still a lower
// bound of the closure. Each changed 16-byte piece is copied into the other
// CTAs (distributed shared memory). Sweep t covers at least the paths of up
// to 2^t edges, so at most ceil(log2 nw) + 1 sweeps run: the cluster stops
// after the first sweep in which no CTA changed anything, when S (x) S <= S
// held for the whole square, i.e. S is closed. Rows of cold candidates are
// zero and stay zero; columns run over all of S. Each CTA then writes its
// rows back into W.
constexpr int kClusterCtas = 8;
constexpr int kClusterThreads = 512;
constexpr int kMaxSweeps = 40;  // > ceil(log2 256) + 1: never reached
constexpr int32_t kSmallMax = 256;  // candidates of closure_small_kernel (kClusterMaxWarm of either lane type)

// acc (16 bytes of a row) = max(acc, min(a(k), b0), min(a(k + 1), b1)) with
// b0, b1 the same 16 bytes of rows k and k + 1 and a the row's entries k,
// k + 1 (one 32-bit word of 16-bit lanes, or an int2)
__device__ __forceinline__ void sweep_step(uint4& acc, uint32_t a, const uint4& b0, const uint4& b1) {
  const uint32_t l = __byte_perm(a, 0, 0x1010), h = __byte_perm(a, 0, 0x3232);
  acc.x = __vimax3_s16x2(acc.x, __vmins2(l, b0.x), __vmins2(h, b1.x));
  acc.y = __vimax3_s16x2(acc.y, __vmins2(l, b0.y), __vmins2(h, b1.y));
  acc.z = __vimax3_s16x2(acc.z, __vmins2(l, b0.z), __vmins2(h, b1.z));
  acc.w = __vimax3_s16x2(acc.w, __vmins2(l, b0.w), __vmins2(h, b1.w));
}
__device__ __forceinline__ void sweep_step(uint4& acc, int2 a, const uint4& b0, const uint4& b1) {
  auto f = [&](uint32_t x, uint32_t u, uint32_t v) {
    return uint32_t(__vimax3_s32(int32_t(x), min(a.x, int32_t(u)), min(a.y, int32_t(v))));
  };
  acc.x = f(acc.x, b0.x, b1.x);
  acc.y = f(acc.y, b0.y, b1.y);
  acc.z = f(acc.z, b0.z, b1.z);
  acc.w = f(acc.w, b0.w, b1.w);
}

__device__ __forceinline__ bool differs(const uint4& a, const uint4& b) {
  return ((a.x ^ b.x) | (a.y ^ b.y) | (a.z ^ b.z) | (a.w ^ b.w)) != 0u;
}

template <typename E>
using RowPair = typename std::conditional<sizeof(E) == 2, uint32_t, int2>::type;  // a row's entries k, k + 1

// One sweep over pieces c0 .. c0 + Q - 1 of the square S4 (rows of Qs 16-byte
// pieces), rows and pivots 0 .. nw - 1 (row nw zero when nw is odd). Returns
// whether the calling thread changed something.
template <typename E>
__device__ __forceinline__ bool sweep_once(cooperative_groups::cluster_group& cl, uint4* S4, int32_t Qs, int32_t c0,
                                           int32_t Q, int32_t nw) {
  using AW = RowPair<E>;
  const AW* A = reinterpret_cast<const AW*>(S4);
  const int32_t ra = Qs * 16 / int32_t(sizeof(AW));  // row stride of A
  const int32_t nwe = (nw + 1) & ~1;                 // pivots, in pairs
  const unsigned q = cl.block_rank();
  const int32_t own = int32_t(q) < nw ? (nw - int32_t(q) + kClusterCtas - 1) / kClusterCtas : 0;
  const int32_t items = (own + 1) / 2 * Q;  // (pair of owned rows, piece)
  bool changed = false;
  for (int32_t it = threadIdx.x; it < items; it += kClusterThreads) {
    const int32_t rp = it / Q, c = c0 + it % Q;
    const int32_t i0 = int32_t(q) + kClusterCtas * (2 * rp), i1 = i0 + kClusterCtas;
    const bool has1 = i1 < nw;
    const uint4 x0 = S4[i0 * Qs + c], x1 = has1 ? S4[i1 * Qs + c] : x0;
    uint4 acc0 = x0, acc1 = x1;
    const AW* a0p = A + i0 * ra;
    const AW* a1p = A + (has1 ? i1 : i0) * ra;
#pragma unroll 4
    for (int32_t k = 0; k < nwe; k += 2) {
      const uint4 b0 = S4[k * Qs + c], b1 = S4[(k + 1) * Qs + c];
      sweep_step(acc0, a0p[k >> 1], b0, b1);
      sweep_step(acc1, a1p[k >> 1], b0, b1);
    }
    if (differs(acc0, x0)) {
      changed = true;
      S4[i0 * Qs + c] = acc0;
#pragma unroll
      for (int o = 1; o < kClusterCtas; ++o) *cl.map_shared_rank(S4 + i0 * Qs + c, (q + o) % kClusterCtas) = acc0;
    }
    if (has1 && differs(acc1, x1)) {
      changed = true;
      S4[i1 * Qs + c] = acc1;
#pragma unroll
      for (int o = 1; o < kClusterCtas; ++o) *cl.map_shared_rank(S4 + i1 * Qs + c, (q + o) % kClusterCtas) = acc1;
    }
  }
  return changed;
}

// Sweeps over the first Q pieces until nothing changes, every copy loaded and
// every flag clear. Returns the number of sweeps.
template <typename E>
__device__ int sweep_square(cooperative_groups::cluster_group& cl, uint4* S4, int32_t Qs, int32_t Q, int32_t nw,
                            uint32_t (*flags)[kClusterCtas]) {
  const int t = threadIdx.x;
  const unsigned q = cl.block_rank();
  int sweeps = 0;
  while (sweeps < kMaxSweeps) {
    const bool changed = sweep_once<E>(cl, S4, Qs, 0, Q, nw);
    ++sweeps;
    const int any = __syncthreads_or(changed);
    if (any && t < kClusterCtas) *cl.map_shared_rank(&flags[sweeps & 1][q], unsigned(t)) = 1u;
    cl.sync();  // this sweep's copies and flags visible everywhere
    const int more = __syncthreads_or(t < kClusterCtas && flags[sweeps & 1][t] != 0u);
    if (t < kClusterCtas) flags[sweeps & 1][t] = 0u;  // rewritten two sweeps on, after the next barrier
    if (!more) break;  // the same decision in every CTA
  }
  return sweeps;
}

template <typename E>
__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(kClusterThreads, 1)
    closure_cluster_kernel(E* __restrict__ W, int32_t ld, const int32_t* __restrict__ warm,
                           unsigned long long* counters) {
  pdl_enter();
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int32_t nw = *warm;
  if (nw == 0 || nw > kClusterMaxWarm<E>) return;  // the same branch in every CTA
  extern __shared__ __align__(16) unsigned char cluster_smem[];
  uint4* S4 = reinterpret_cast<uint4*>(cluster_smem);
  __shared__ uint32_t flags[2][kClusterCtas];     // CTA o changed something in the sweep (two buffers)
  const int32_t n = (nw + kB - 1) / kB * kB;      // square side: whole 64-wide tiles
  constexpr int kPer16 = 16 / sizeof(E);          // entries per 16-byte piece
  const int32_t Q = n / kPer16;                   // pieces per row
  const int32_t nwe = (nw + 1) & ~1;              // pivots, in pairs (row nw, if read, is zero)
  const int t = threadIdx.x;
  const unsigned q = cl.block_rank();
  {
    // rows 0 .. nwe - 1 of W, eight 16-byte loads in flight per thread
    const int32_t total = nwe * Q;
    constexpr int kU = 8;
    for (int32_t e0 = t; e0 < total; e0 += kU * kClusterThreads) {
      uint4 v[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int32_t e = e0 + u * kClusterThreads;
        if (e < total) v[u] = __ldcg(reinterpret_cast<const uint4*>(W + int64_t(e / Q) * ld) + e % Q);
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int32_t e = e0 + u * kClusterThreads;
        if (e < total) S4[e] = v[u];
      }
    }
  }
  if (t < 2 * kClusterCtas) flags[t / kClusterCtas][t % kClusterCtas] = 0u;
  cl.sync();  // every copy loaded, every flag clear, before any remote write
  const int32_t own = int32_t(q) < nw ? (nw - int32_t(q) + kClusterCtas - 1) / kClusterCtas : 0;
  const int sweeps = sweep_square<E>(cl, S4, Q, Q, nw, flags);
  // each CTA writes its rows back with a zero diagonal. No CTA writes into
  // another any more.
  for (int32_t it = t; it < own * Q; it += kClusterThreads) {
    const int32_t r = it / Q, c = it % Q;
    const int32_t i = int32_t(q) + kClusterCtas * r, j0 = c * kPer16;
    uint4 v = S4[i * Q + c];
    if (i >= j0 && i < j0 + kPer16) {
      const int e = i - j0;
      const int w = sizeof(E) == 2 ? e >> 1 : e;
      const uint32_t keep = sizeof(E) == 2 ? ((e & 1) ? 0x0000FFFFu : 0xFFFF0000u) : 0u;
      v.x = w == 0 ? v.x & keep : v.x;
      v.y = w == 1 ? v.y & keep : v.y;
      v.z = w == 2 ? v.z & keep : v.z;
      v.w = w == 3 ? v.w & keep : v.w;
    }
    *reinterpret_cast<uint4*>(W + int64_t(i) * ld + j0) = v;
  }
  if (t == 0 && q == 0)  // entry updates, in 64 x 64 x 64 tile units
    atomicAdd(&counters[0], (unsigned long long)sweeps * uint64_t(nw) * uint64_t(nw) * uint64_t(n) / 262144ull);
}

// Elections of at most kClusterMaxWarm candidates: the whole way from d to p,
// beaten_by, winners and order in one launch of the cluster (each of bb,
// winners and order may be null). CTA q makes the weights of rows q, q + 8,
// ... (eight entries per thread: 32 bytes of the row, and the transposed
// column) and copies them into every CTA's square, rows one 16-byte piece
// longer than they need so that a column's entries spread over the banks;
// after the sweeps it writes its rows of p, counts who beats its candidates,
// hands the counts to the other CTAs and ranks its candidates. Bound by
// latency: it replaces a chain of eleven launches (m = 64: 10 us).
//
// From kFewMin on, where enough candidates have no edge, the square is filled
// anew with those that have one first (the other rows are zero and are left out,
// as pivots too), the sweeps run over it alone and one more takes its widths to
// the other columns: m = 256, int16: 5% with edges 81 -> 27 us, 50% 117 -> 50, 80%
// 120 -> 100; m = 192, int32: 70 -> 22, 103 -> 45, 106 -> 84. The second filling
// takes 2 to 4 us. What it saves grows with the entries of the rows left out: at
// m = 150, int32, 15 rows are about even (56.1 and 58.3 us), 22 save 7 us. Up to
// 128 candidates, where all of them take no more than 38 us, looking for edges
// costs more than it saves (m = 64: 15.4 and 15.9 us, all with edges).
constexpr int32_t kFewMin = 129, kFewSaving = 2400;
template <typename E>
__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(kClusterThreads, 1)
    closure_small_kernel(const int32_t* __restrict__ d, int32_t m, int64_t bound, int margin, int32_t* __restrict__ p,
                         int32_t* __restrict__ bb, int32_t* __restrict__ winners, int32_t* __restrict__ order,
                         int32_t* status, unsigned long long* counters) {
  pdl_enter();
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char small_smem[];
  constexpr int kPer16 = 16 / sizeof(E);
  const int32_t Q = (m + kPer16 - 1) / kPer16, Qs = Q + 1;
  uint4* S4 = reinterpret_cast<uint4*>(small_smem);
  const E* S = reinterpret_cast<const E*>(small_smem);  // entry (i, j): S[i * ls + j]
  const int32_t ls = Qs * kPer16;
  __shared__ uint32_t flags[2][kClusterCtas];
  __shared__ int32_t beaten[kSmallMax];
  __shared__ uint8_t edges[kSmallMax];               // whether candidate i has an edge
  __shared__ uint16_t perm[kSmallMax], pos[kSmallMax];  // those with one first: new -> old, old -> new
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const unsigned q = cl.block_rank();
  const int32_t own = int32_t(q) < m ? (m - int32_t(q) + kClusterCtas - 1) / kClusterCtas : 0;
  if (t < 2 * kClusterCtas) flags[t / kClusterCtas][t % kClusterCtas] = 0u;
  if (t < kSmallMax) edges[t] = 0;
  if (m & 1)  // the row past the last one, which a pair of pivots reads
    for (int32_t c = t; c < Q; c += kClusterThreads) S4[m * Qs + c] = make_uint4(0u, 0u, 0u, 0u);
  cl.sync();  // every CTA has started before any remote write
  bool bad = false;
  // the weights of n of this CTA's rows into every square, candidate(x) in its row or column x
  auto fill = [&](int32_t n, auto candidate) {
    for (int32_t it = t; it < n * Q; it += kClusterThreads) {
      const int32_t c = it / n, a = int32_t(q) + kClusterCtas * (it - c * n), i = candidate(a), j0 = c * kPer16;
      int32_t x[kPer16], y[kPer16];
#pragma unroll
      for (int e = 0; e < kPer16; ++e) {
        const int32_t j = j0 + e < m ? candidate(j0 + e) : 0;
        x[e] = j0 + e < m ? d[int64_t(i) * m + j] : 0;
        y[e] = j0 + e < m ? d[int64_t(j) * m + i] : 0;
      }
      uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int e = 0; e < kPer16; ++e) {
        bad |= x[e] < 0 || int64_t(x[e]) > bound;
        const int32_t out = x[e] > y[e] ? x[e] - (margin ? y[e] : 0) : 0;
        if (sizeof(E) == 2) w[e >> 1] |= (uint32_t(out) & 0xFFFFu) << (16 * (e & 1));
        else w[e & 3] = uint32_t(out);
      }
      const uint4 v = make_uint4(w[0], w[1], w[2], w[3]);
      if (v.x | v.y | v.z | v.w) edges[i] = 1;
#pragma unroll
      for (int o = 0; o < kClusterCtas; ++o) *cl.map_shared_rank(S4 + a * Qs + c, unsigned(o)) = v;
    }
  };
  fill(own, [](int32_t x) { return x; });
  if (bad) set_status(status, SCHULZE_EDATA);
  const bool look = m >= kFewMin;
  if (look) {  // the own candidates' edges, told to the others
    __syncthreads();
    for (int x = t; x < own * kClusterCtas; x += kClusterThreads) {
      const int32_t i = int32_t(q) + kClusterCtas * (x / kClusterCtas), o = x % kClusterCtas;
      if (o != int32_t(q)) *cl.map_shared_rank(edges + i, unsigned(o)) = edges[i];
    }
  }
  cl.sync();  // every square and edge list complete
  int32_t nw = m;
  if (look) {
    nw = __syncthreads_count(t < m && edges[t]);
    if ((m - nw) * m < kFewSaving) nw = m;
  }
  const bool few = nw < m;  // (the same decision in every CTA)
  int sweeps;
  if (few) {
    if (wid == 0) {
      int32_t seen = 0;  // candidates with edges so far
      for (int32_t i0 = 0; i0 < m; i0 += 32) {
        const int32_t i = i0 + lane;
        const uint32_t b = __ballot_sync(0xFFFFFFFFu, i < m && edges[i]);
        const int32_t before = seen + __popc(b & ((1u << lane) - 1u));
        if (i < m) {
          const int32_t a = edges[i] ? before : nw + i - before;
          pos[i] = uint16_t(a), perm[a] = uint16_t(i);
        }
        seen += __popc(b);
      }
    }
    if (nw & 1)
      for (int32_t c = t; c < Q; c += kClusterThreads) S4[nw * Qs + c] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();  // (no CTA reads its square before the next cluster barrier)
    fill(int32_t(q) < nw ? (nw - int32_t(q) + kClusterCtas - 1) / kClusterCtas : 0,
         [&](int32_t x) { return int32_t(perm[x]); });
    cl.sync();
    const int32_t Qw = (nw + kPer16 - 1) / kPer16;
    sweeps = sweep_square<E>(cl, S4, Qs, Qw, nw, flags);
    if (Qw < Q) {
      sweep_once<E>(cl, S4, Qs, Qw, Q - Qw, nw);
      cl.sync();
    }
  } else {
    sweeps = sweep_square<E>(cl, S4, Qs, Q, m, flags);
  }
  auto rows_out = [&](auto width) {  // width(i, j), i != j
    for (int32_t r = wid; r < own; r += kClusterThreads / 32) {
      const int32_t i = int32_t(q) + kClusterCtas * r;
      int32_t c = 0;
      for (int32_t j = lane; j < m; j += 32) {
        const int32_t x = j == i ? 0 : width(i, j);
        p[int64_t(i) * m + j] = x;
        c += j != i && width(j, i) > x;
      }
      c = __reduce_add_sync(0xFFFFFFFFu, c);
      if (lane < kClusterCtas) *cl.map_shared_rank(beaten + i, unsigned(lane)) = c;
    }
  };
  if (few) rows_out([&](int32_t i, int32_t j) { return edges[i] ? int32_t(S[pos[i] * ls + pos[j]]) : 0; });
  else rows_out([&](int32_t i, int32_t j) { return int32_t(S[i * ls + j]); });
  cl.sync();  // every count everywhere
  for (int32_t r = wid; r < own; r += kClusterThreads / 32) {
    const int32_t i = int32_t(q) + kClusterCtas * r, count = beaten[i];
    int32_t ahead = 0;  // candidates ahead of i by (beaten_by, id)
    for (int32_t j = lane; j < m; j += 32) ahead += beaten[j] < count || (beaten[j] == count && j < i);
    ahead = __reduce_add_sync(0xFFFFFFFFu, ahead);
    if (lane == 0) {
      if (bb) bb[i] = count;
      if (winners) winners[i] = count == 0;
      if (order) order[ahead] = i;
    }
  }
  if (t == 0 && q == 0)  // entry updates, in 64 x 64 x 64 tile units
    atomicAdd(&counters[0], (unsigned long long)sweeps * uint64_t(nw) * uint64_t(nw) * uint64_t(nw) / 262144ull);
}

// Uniform cold columns: u[i] = max(ucol[i], max_x min(W[i][x], ucol[x]))
// over the warm x (a warp per warm row i, lanes over x), and ucount = the
// number of warm rows with u > 0.
template <typename E>
__global__ void __launch_bounds__(256) uniform_cold_kernel(const E* __restrict__ W, int32_t mp, int32_t m,
                                                           const int32_t* __restrict__ warm,
                                                           const int32_t* __restrict__ hint_valid,
                                                           const int32_t* __restrict__ ucol, int32_t* __restrict__ u,
                                                           int32_t* __restrict__ ucount) {
  pdl_enter();
  const int32_t nw = *warm;
  const int32_t rows = (nw + kB - 1) / kB * kB;
  if (!(hint_valid && *hint_valid && rows < m)) return;
  const int lane = threadIdx.x & 31;
  const int64_t wid = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t i = wid; i < nw; i += nwarps) {
    const E* wrow = W + i * mp;
    int32_t best = 0;
    for (int32_t x = lane; x < nw; x += 32) best = max(best, min(int32_t(wrow[x]), ucol[x]));
#pragma unroll
    for (int o = 16; o; o >>= 1) best = max(best, __shfl_xor_sync(0xFFFFFFFFu, best, o));
    if (lane == 0) {
      const int32_t ui = max(best, ucol[i]);
      u[i] = ui;
      if (ui > 0) atomicAdd(ucount, 1);
    }
  }
}

// Cold columns for warm squares that fit shared memory (the cluster
// closure's sizes): every CTA keeps the closed square P (nwp x nwp, rows
// padded by one word against bank conflicts) and walks strips of
// kStripWords words (16-bit pairs, or int32 entries) of cold columns:
// X[i][j] = max(X[i][j], max_k min(P[i][k], X[k][j])) for the warm rows i,
// with X[k][j] staged before any row of the strip is written. Thread t keeps
// words w and w + 8 (w = t % 8) of rows t / 8 + 64 r, r < 4, so that each
// load of P or of the strip feeds several updates.
constexpr int kStripWords = 16;

template <typename E>
__global__ void __launch_bounds__(512, 1) cold_strip_kernel(E* __restrict__ W, int32_t ld, int32_t m,
                                                            const int32_t* __restrict__ warm,
                                                            unsigned long long* counters,
                                                            const int32_t* __restrict__ hint_valid) {
  // With a hint cold_product_kernel seldom has work; without one its CTAs are
  // let in late, when they spread over SMs that the closure has left
  if (hint_valid) pdl_enter_early();
  else pdl_enter();
  using Wd = typename std::conditional<sizeof(E) == 2, uint32_t, int32_t>::type;  // one word
  constexpr int kPer = sizeof(Wd) / sizeof(E);                                  // entries per word
  const int32_t nw = *warm;
  if (nw == 0 || nw > kClusterMaxWarm<E>) return;  // the tile kernel's case
  const int32_t nwp = (nw + kB - 1) / kB * kB;
  if (hint_valid && *hint_valid && nwp < m) return;  // uniform cold columns
  const int32_t rowwords = ld / kPer;
  const int32_t nstrips = (rowwords - nwp / kPer + kStripWords - 1) / kStripWords;
  if (int32_t(blockIdx.x) >= nstrips) return;
  extern __shared__ __align__(16) unsigned char strip_smem[];
  const int32_t pw = nwp / kPer, pst = pw + 1;  // words per row of P, padded (odd)
  Wd* P = reinterpret_cast<Wd*>(strip_smem);
  Wd* B = P + nwp * pst;  // [nwp][kStripWords]
  const int t = threadIdx.x;
  for (int32_t e = t; e < nwp * (pw / 4); e += blockDim.x) {  // 16-byte reads of W
    const int32_t i = e / (pw / 4), c4 = e % (pw / 4);
    const uint4 v = __ldcg(reinterpret_cast<const uint4*>(W + int64_t(i) * ld) + c4);
    Wd* dst = P + i * pst + 4 * c4;
    dst[0] = Wd(v.x), dst[1] = Wd(v.y), dst[2] = Wd(v.z), dst[3] = Wd(v.w);
  }
  const int w = t & 7, rg = t >> 3;  // words w, w + 8; rows rg + 64 r
  const int32_t K = (nw + 1) & ~1;   // rows >= nw are zero
  unsigned long long done = 0;
  for (int32_t s = blockIdx.x; s < nstrips; s += gridDim.x) {
    const int32_t c0 = pw + s * kStripWords;  // first word of the strip
    __syncthreads();  // P loaded / the previous strip's B consumed
    for (int32_t e = t; e < nwp * kStripWords; e += blockDim.x) {
      const int32_t k = e / kStripWords, c = c0 + e % kStripWords;
      B[e] = c < rowwords ? reinterpret_cast<const Wd*>(W + int64_t(k) * ld)[c] : Wd(0);
    }
    __syncthreads();
    Wd acc[4][2];
    bool row_ok[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int32_t i = rg + 64 * r;
      row_ok[r] = i < nw;
      acc[r][0] = row_ok[r] ? B[i * kStripWords + w] : Wd(0);
      acc[r][1] = row_ok[r] ? B[i * kStripWords + w + 8] : Wd(0);
    }
#pragma unroll 2
    for (int32_t k = 0; k < K; k += 2) {
      const Wd b00 = B[k * kStripWords + w], b01 = B[k * kStripWords + w + 8];
      const Wd b10 = B[(k + 1) * kStripWords + w], b11 = B[(k + 1) * kStripWords + w + 8];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (!row_ok[r]) continue;
        const Wd* prow = P + (rg + 64 * r) * pst;
        if constexpr (sizeof(E) == 2) {
          const uint32_t a = prow[k >> 1];
          const uint32_t alo = (a & 0xFFFFu) | (a << 16), ahi = (a >> 16) | (a & 0xFFFF0000u);
          acc[r][0] = __vimax3_s16x2(acc[r][0], __vmins2(alo, b00), __vmins2(ahi, b10));
          acc[r][1] = __vimax3_s16x2(acc[r][1], __vmins2(alo, b01), __vmins2(ahi, b11));
        } else {
          const int32_t a0 = prow[k], a1 = prow[k + 1];
          acc[r][0] = __vimax3_s32(acc[r][0], min(a0, b00), min(a1, b10));
          acc[r][1] = __vimax3_s32(acc[r][1], min(a0, b01), min(a1, b11));
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (!row_ok[r]) continue;
      Wd* dst = reinterpret_cast<Wd*>(W + int64_t(rg + 64 * r) * ld) + c0;
      if (c0 + w < rowwords) dst[w] = acc[r][0];
      if (c0 + w + 8 < rowwords) dst[w + 8] = acc[r][1];
    }
    ++done;
  }
  if (t == 0 && done) atomicAdd(&counters[0], done);
}

// Cold columns: X(i, j) = max(X, W(i, k) (x) W(k, j)) for every warm tile row
// i, cold tile column j and warm k, with the warm square already closed. Each
// (i, j) is one work item (a 128-thread CTA applies its k in order). An item
// may read a W(k, j) that another item is raising at the same time; every
// value either one sees is the width of a real path and the closed square
// composes with itself without growing (p(i,x) and p(x,y) give a walk no
// wider than p(i,y)), so the result is the exact closure either way. Five CTAs
// per SM (without the bound 32-bit lanes take registers for three), launched
// once the closure is done (cold_strip_kernel) where there is no hint: m = 8192
// with 3000 warm, int32, the whole call 8.32 -> 7.83 ms; with the bound alone 7.80,
// but m = 2000 with 1000 0.73 -> 0.85 then, as CTAs that came early took the SMs
// unevenly. (Seven CTAs with 16-bit lanes: 1% less here, and 0.5 us more where
// they return at once.)
template <typename E>
__global__ void __launch_bounds__(kThreads, 5)
    cold_product_kernel(E* __restrict__ W, int32_t ld, int32_t nb, int32_t m, const int32_t* __restrict__ warm,
                        const unsigned long long* __restrict__ prog, const int32_t* __restrict__ tmax,
                        unsigned long long* counters, const int32_t* __restrict__ hint_valid) {
  pdl_enter_early();
  __shared__ __align__(16) typename Ops<E>::Smem sm;
  if (*warm <= kClusterMaxWarm<E>) return;  // cold_strip_kernel's case
  if (hint_valid && *hint_valid && (*warm + kB - 1) / kB * kB < m) return;  // uniform cold columns
  const int32_t nbr = (*warm + kB - 1) / kB;
  const int32_t nc = nb - nbr;
  const int64_t items = int64_t(nbr) * nc;
  unsigned long long done = 0;
  for (int64_t t = blockIdx.x; t < items; t += gridDim.x) {
    const int32_t i = int32_t(t / nc), j = nbr + int32_t(t % nc);
    for (int32_t k = 0; k < nbr; ++k) {
      if (word_max(prog[i * nb + k]) && tmax[k * nb + j]) {  // both operands hold a nonzero
        tiles::tile_update(W, ld, i, j, k, sm, threadIdx.x, BlockBarrier{});
        ++done;
      }
    }
  }
  if (threadIdx.x == 0 && done) atomicAdd(&counters[0], done);
}

// beaten_by straight from the closed warm rows of W, for callers that need
// the ranking but not a second pass over p: a cold candidate x (no outgoing
// edge, p[x][*] = 0) is beaten by every warm j with p[j][x] > 0; a warm x by
// every warm j with p[j][x] > p[x][j]; cold candidates beat nobody.
//
// Squares of the persistent closure: CTA (J, c) counts, for the 64 columns of
// tile column J, the rows of tile rows 32 c .. 32 c + 31 that beat them, and
// adds the counts into bb (zeroed before). The tiles' bounds in the progress
// words decide most pairs of tiles unread (every width of (I, J) above every
// width of (J, I), or none): in strength order that is all but the ones near
// the diagonal (m = 16384, int32: 0.086 ms, against 1.25 ms reading all of W).
// Smaller squares: CTA = 32 relabeled columns x 16 row groups.
template <typename E>
__global__ void __launch_bounds__(512) wextract_kernel(const E* __restrict__ W, int32_t mp, int32_t m,
                                                       const int32_t* __restrict__ perm,
                                                       const int32_t* __restrict__ warm, int32_t* __restrict__ bb,
                                                       const int32_t* __restrict__ hint_valid,
                                                       const int32_t* __restrict__ ucount,
                                                       const unsigned long long* __restrict__ prog, int32_t nb,
                                                       int32_t warm_max) {
  pdl_enter();
  constexpr int kG = 16;  // row groups
  __shared__ int32_t part[kG][33];
  const int32_t nw = *warm;
  const int32_t rows = (nw + kB - 1) / kB * kB;
  const bool uc = hint_valid && *hint_valid && rows < m;
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  if (nw > warm_max) {
    __shared__ E tj[kB][kB + (sizeof(E) == 2 ? 2 : 1)];  // tile (J, I), rows an odd number of words apart
    __shared__ int32_t cnt[kB];
    __shared__ uint32_t s_read;
    const int32_t nbr = rows / kB, nchunk = (nbr + 31) / 32;
    for (int32_t t = blockIdx.x; t < nb * nchunk; t += gridDim.x) {
      const int32_t J = t / nchunk, I0 = (t - J * nchunk) * 32;
      if (uc && J >= nbr) {  // uniform cold columns: beaten by the warm rows with u > 0
        if (I0 == 0 && threadIdx.x < kB && J * kB + int32_t(threadIdx.x) < m)
          bb[perm[J * kB + threadIdx.x]] = *ucount;
        continue;
      }
      if (g == 0) {  // warp 0 alone starts every counter, before the barrier
        // all: every row of tile (I, J) with edges beats every column; none:
        // no row beats any (cold columns, whose own rows are zero, need the
        // tile itself to be zero)
        const int32_t I = I0 + lane;
        int32_t all = 0;
        bool read = false;
        if (I < nbr) {
          const bool warm_j = J < nbr, cold_in_j = (J + 1) * kB > nw;
          const uint64_t wij = warm_j ? prog[I * nb + J] : 0, wji = warm_j ? prog[J * nb + I] : 0;
          if (I != J && warm_j && word_min(wij) > word_max(wji)) all = min(kB, nw - I * kB);
          else read = !warm_j || I == J || (cold_in_j ? word_max(wij) > 0 : word_max(wij) > word_min(wji));
        }
        const uint32_t mask = __ballot_sync(0xFFFFFFFFu, read);
        all = __reduce_add_sync(0xFFFFFFFFu, all);
        if (lane == 0) s_read = mask;
        __syncwarp();
        cnt[lane] = all, cnt[lane + 32] = all;
      }
      __syncthreads();
      int32_t c = 0;
      const int col = threadIdx.x & (kB - 1), rg = threadIdx.x / kB;  // column, rows rg + 8 q
      for (uint32_t mask = s_read; mask; mask &= mask - 1) {
        const int32_t I = I0 + __ffs(int(mask)) - 1;
        for (int e = threadIdx.x; e < kB * kB; e += blockDim.x) {  // (rows past the square are not in W)
          const int32_t j = J * kB + e / kB;
          tj[e / kB][e % kB] = j < rows ? W[int64_t(j) * mp + I * kB + e % kB] : E(0);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kB / 8; ++q) {
          const int i = rg + 8 * q;
          const bool in = I * kB + i < nw && J * kB + col < m && !(I == J && i == col);
          if (in) c += int32_t(W[int64_t(I * kB + i) * mp + J * kB + col]) > int32_t(tj[col][i]);
        }
        __syncthreads();
      }
      if (c) atomicAdd(&cnt[col], c);
      __syncthreads();
      if (threadIdx.x < kB && J * kB + int32_t(threadIdx.x) < m && cnt[threadIdx.x])
        atomicAdd(&bb[perm[J * kB + threadIdx.x]], cnt[threadIdx.x]);
      __syncthreads();
    }
    return;
  }
  for (int32_t b0 = blockIdx.x * 32; b0 < m; b0 += gridDim.x * 32) {
    if (uc && b0 >= rows) {  // uniform cold columns: beaten by the warm rows with u > 0
      if (g == 0 && b0 + lane < m) bb[perm[b0 + lane]] = *ucount;
      continue;
    }
    const int32_t b = b0 + lane;
    int32_t c = 0;
    if (b < m) {
      if (b < nw) {
#pragma unroll 4
        for (int32_t j = g; j < nw; j += kG)
          c += (j != b && int32_t(W[int64_t(j) * mp + b]) > int32_t(W[int64_t(b) * mp + j]));
      } else {
#pragma unroll 8
        for (int32_t j = g; j < nw; j += kG) c += W[int64_t(j) * mp + b] != E(0);
      }
    }
    part[g][lane] = c;
    __syncthreads();
    if (g == 0 && b < m) {
      int32_t tot = 0;
#pragma unroll
      for (int h = 0; h < kG; ++h) tot += part[h][lane];
      bb[perm[b]] = tot;
    }
    __syncthreads();
  }
}

// Scratch of one closure: W (warm rows x all columns, padded square), the
// progress words, queue head, abort flag, and the relabeling.
struct ClosureBufs {
  void* W;
  uint32_t* prog;  // prog_words(nb): progress words, packed tiles' bounds, queue head, abort flag
  int32_t *rowflag, *perm, *inv, *warm;
  unsigned long long* counters;
  // optional: warm flags known from the tally, used when *hint_valid != 0
  const int32_t* hint = nullptr;
  const int32_t* hint_valid = nullptr;
  // uniform cold columns (used only with a valid hint): ucol, u [m], ucount
  int32_t *ucol = nullptr, *ucold = nullptr, *ucount = nullptr;
  bool margin = false;  // margin weights instead of winning votes
  bool zeroed = false;  // prog, rowflag, ucount and beaten_by are zero already
};

constexpr size_t prog_words(size_t nb) { return 4 * nb * nb + 2; }
constexpr size_t kMaxRowBuf = 200 * 1024;  // larger rows (int32, m > 51200) are gathered from global memory

// Rowflags, relabel, pack, closure of the warm square, cold product, widen.
// ctx may be null (no counting, no profiling).
template <typename E>
int closure_pipeline(schulze_ctx* ctx, int sms, const int32_t* d, int32_t m, int64_t bound, int32_t* p,
                     const ClosureBufs& bf, int32_t* status, cudaStream_t stream, int32_t* bb_out = nullptr,
                     bool side = false, int32_t* winners = nullptr, int32_t* order = nullptr) {
  if (m <= kClusterMaxWarm<E>) {
    constexpr int kPer16 = 16 / int(sizeof(E));
    const size_t Q = size_t(m + kPer16 - 1) / kPer16, smem = size_t(m + 1) * (Q + 1) * 16;
    raise_smem(ctx, reinterpret_cast<const void*>(closure_small_kernel<E>));
    Launch L(ctx, stream, "closure_small", double(m) * double(m) * double(m));
    launch_pdl(closure_small_kernel<E>, dim3(kClusterCtas), dim3(kClusterThreads), smem, stream, false, d, m, bound,
               bf.margin ? 1 : 0, p, bb_out, winners, order, status, bf.counters);
    return check_launch();
  }
  const int32_t mp = int32_t(align_up(size_t(m), kB));
  const int32_t nb = mp / kB;
  E* W = static_cast<E*>(bf.W);
  const Weights<E> V = weights_in<E>(p, m);
  const size_t tiles2 = size_t(nb) * size_t(nb);
  unsigned long long* prog = reinterpret_cast<unsigned long long*>(bf.prog);
  int32_t* tmax = reinterpret_cast<int32_t*>(bf.prog + 2 * tiles2);
  int32_t* tmin = tmax + tiles2;
  uint32_t* head = bf.prog + 4 * tiles2;
  uint32_t* abort_flag = head + 1;
  const int shift = word_shift(bound);
  if (!bf.zeroed) {
    // progress words, tile bounds, queue head and abort flag; row flags; the uniform count
    ZeroSpans z;
    z.add(bf.prog, int64_t(prog_words(size_t(nb)))), z.add(bf.rowflag, m), z.add(bf.ucount, 1), z.add(bb_out, m);
    if (int rc = zero_async(ctx, z, stream)) return rc;
  }
  const double mm = double(m) * double(m);
  auto grid_for = [&](const void* fn, int threads, size_t smem, int64_t cap) {
    const int per_sm = blocks_per_sm(ctx, fn, threads, smem);
    return int(std::max<int64_t>(1, std::min<int64_t>(int64_t(per_sm) * sms, cap)));
  };
  {
    const int64_t nbt = (m + kFlagT - 1) / kFlagT;
    auto kern = bf.margin ? weigh_kernel<E, true> : weigh_kernel<E, false>;
    const int g = grid_for(reinterpret_cast<const void*>(kern), 256, 0, nbt * (nbt + 1) / 2);
    Launch L(ctx, stream, "closure_rowflags", mm * 4.0);
    launch_pdl(kern, dim3(g), dim3(256), 0, stream, false, d, m, bound, bf.rowflag, status,
               static_cast<const int32_t*>(bf.warm), bf.hint_valid, kClusterMaxWarm<E>, rows_vec16(d, m), V);
  }
  {
    Launch L(ctx, stream, "closure_relabel", double(m) * 12.0);
    const size_t smem = m <= kScanSmem ? size_t(m) * 4 : 0;
    raise_smem(ctx, reinterpret_cast<const void*>(relabel_kernel));
    launch_pdl(relabel_kernel, dim3(1), dim3(1024), smem, stream, false,
               static_cast<const int32_t*>(bf.rowflag), m, bf.perm, bf.inv, bf.warm, bf.hint, bf.hint_valid,
               kClusterMaxWarm<E>);
  }
  // rows of the weights and of W in shared memory, up to what a CTA can have
  const size_t rowbytes = align_up(size_t(mp) * sizeof(E), 16);
  const uint32_t rowbuf = rowbytes <= kMaxRowBuf ? uint32_t(rowbytes) : 0u;
  {
    const size_t smem = rowbuf + 2 * size_t(nb) * 4;
    const int32_t chunk = m >= 8192 ? 16 : m >= 2048 ? 4 : 1;
    raise_smem(ctx, reinterpret_cast<const void*>(pack_kernel<E>));
    const int g = grid_for(reinterpret_cast<const void*>(pack_kernel<E>), 512, smem, mp);
    Launch L(ctx, stream, "closure_pack", 0.0);
    launch_pdl(pack_kernel<E>, dim3(g), dim3(512), smem, stream, false, d, m, mp,
               static_cast<const int32_t*>(bf.perm), static_cast<const int32_t*>(bf.warm), W, tmax, tmin, nb, bf.hint,
               bf.hint_valid, bf.ucol, bf.margin ? 1 : 0, kClusterMaxWarm<E>, V, rowbuf, chunk);
  }
  if (int rc = check_launch()) return rc;
  {
    const size_t smem = size_t(kClusterMaxWarm<E>) * kClusterMaxWarm<E> * sizeof(E);
    raise_smem(ctx, reinterpret_cast<const void*>(closure_cluster_kernel<E>));
    Launch L(ctx, stream, "closure_cluster", 0.0);
    launch_pdl(closure_cluster_kernel<E>, dim3(kClusterCtas), dim3(kClusterThreads), smem, stream, false, W, mp,
               static_cast<const int32_t*>(bf.warm), bf.counters);
  }
  if (int rc = check_launch()) return rc;
  {
    // persistent grid: every CTA resident (cooperative launch)
    const int grid = grid_for(reinterpret_cast<const void*>(closure_persistent_kernel<E>), kThreads, 0,
                              int64_t(nb) * nb * nb);
    Sync sy{prog, tmax, tmin, head, abort_flag, status, bf.warm, bf.counters,
            ctx ? ctx->wait_limit_cycles : kSpinLimitCycles, shift};
    Launch L(ctx, stream, "closure_persistent", double(m) * mm);
    if (launch_pdl(closure_persistent_kernel<E>, dim3(grid), dim3(kThreads), 0, stream, true, W, mp, m, nb, sy) !=
        cudaSuccess) {
      cudaGetLastError();
      return SCHULZE_ECUDA;
    }
  }
  {
    const size_t cw = size_t(kClusterMaxWarm<E>);
    const size_t smem = (cw * (cw * sizeof(E) / 4 + 1) + cw * kStripWords) * 4;
    raise_smem(ctx, reinterpret_cast<const void*>(cold_strip_kernel<E>));
    Launch L(ctx, stream, "closure_cold_strips", 0.0);
    launch_pdl(cold_strip_kernel<E>, dim3(sms), dim3(512), smem, stream, false, W, mp, m,
               static_cast<const int32_t*>(bf.warm), bf.counters, bf.hint_valid);
  }
  {
    const int g = grid_for(reinterpret_cast<const void*>(cold_product_kernel<E>), kThreads, 0, int64_t(nb) * nb);
    Launch L(ctx, stream, "closure_cold", 0.0);
    launch_pdl(cold_product_kernel<E>, dim3(g), dim3(kThreads), 0, stream, false, W, mp, nb, m,
               static_cast<const int32_t*>(bf.warm), static_cast<const unsigned long long*>(prog),
               static_cast<const int32_t*>(tmax), bf.counters, bf.hint_valid);
  }
  if (bf.hint_valid) {
    Launch L(ctx, stream, "closure_cold_uniform", 0.0);
    launch_pdl(uniform_cold_kernel<E>, dim3(std::max(1, std::min(sms, (m + 7) / 8))), dim3(256), 0, stream, false,
               static_cast<const E*>(W), mp, m, static_cast<const int32_t*>(bf.warm), bf.hint_valid,
               static_cast<const int32_t*>(bf.ucol), bf.ucold, bf.ucount);
  }
  {
    // p is written from W (and the uniform cold values); with a side stream
    // it is written there while beaten_by and the ranking come out of W on
    // stream, with at most two CTAs per SM so that those kernels find room
    const bool fork = side && bb_out && ctx && ctx->side_stream;
    cudaStream_t wst = stream;
    raise_smem(ctx, reinterpret_cast<const void*>(widen_kernel<E>));
    int g = grid_for(reinterpret_cast<const void*>(widen_kernel<E>), 512, rowbuf, m);
    if (fork) {
      if (cudaEventRecord(ctx->side_fork, stream) != cudaSuccess ||
          cudaStreamWaitEvent(ctx->side_stream, ctx->side_fork, 0) != cudaSuccess)
        return SCHULZE_ECUDA;
      ctx->side_pending = true;  // joined by the caller, whatever happens next
      wst = ctx->side_stream;
      g = std::min(g, 2 * sms);
    }
    Launch L(ctx, wst, "closure_widen", mm * 4.0);
    launch_pdl(widen_kernel<E>, dim3(g), dim3(512), rowbuf, wst, false, static_cast<const E*>(W), mp, m,
               static_cast<const int32_t*>(bf.inv), static_cast<const int32_t*>(bf.perm),
               static_cast<const int32_t*>(bf.warm), p, bf.hint_valid, static_cast<const int32_t*>(bf.ucold),
               rows_vec16(p, m), rowbuf);
    if (fork && cudaEventRecord(ctx->side_join, wst) != cudaSuccess) return SCHULZE_ECUDA;
  }
  if (bb_out) {
    Launch L(ctx, stream, "closure_beaten_by", 0.0);
    launch_pdl(wextract_kernel<E>, dim3((m + 31) / 32), dim3(512), 0, stream, false, static_cast<const E*>(W), mp, m,
               static_cast<const int32_t*>(bf.perm), static_cast<const int32_t*>(bf.warm), bb_out, bf.hint_valid,
               static_cast<const int32_t*>(bf.ucount), static_cast<const unsigned long long*>(prog), nb,
               kClusterMaxWarm<E>);
  }
  return check_launch();
}

template <typename E>
int run_closure(schulze_ctx* ctx, const int32_t* d, int32_t m, int64_t bound, int32_t* p, void* ws,
                cudaStream_t stream, int32_t* bb_out, int32_t* hint, const int32_t* hint_valid,
                bool margin, bool side, int32_t* winners, int32_t* order, uint32_t* control) {
  const int32_t mp = int32_t(align_up(size_t(m), kB));
  const int32_t nb = mp / kB;
  Carver cv(ws);
  ClosureBufs bf;
  bf.W = cv.take<E>(size_t(mp) * size_t(mp));
  bf.prog = cv.take<uint32_t>(prog_words(size_t(nb)));
  bf.rowflag = cv.take<int32_t>(size_t(m));
  bf.perm = cv.take<int32_t>(size_t(m));
  bf.inv = cv.take<int32_t>(size_t(m));
  bf.warm = cv.take<int32_t>(1);
  if (hint) {  // the relabeling lives with the tally's flags (written there when they are valid)
    bf.perm = hint + m;
    bf.inv = hint + 2 * size_t(m);
    bf.warm = hint + 3 * size_t(m);
  }
  bf.ucol = cv.take<int32_t>(size_t(m));
  bf.ucold = cv.take<int32_t>(size_t(m));
  bf.ucount = cv.take<int32_t>(1);
  if (control) {  // (closure_control_words)
    bf.prog = control;
    bf.rowflag = reinterpret_cast<int32_t*>(control + prog_words(size_t(nb)));
    bf.ucount = bf.rowflag + m;
    bf.zeroed = true;
  }
  bf.counters = ctx->counters;
  bf.hint = hint;
  bf.hint_valid = hint_valid;
  bf.margin = margin;
  const int sms = ctx->sm_count > 0 ? ctx->sm_count : 1;
  return closure_pipeline<E>(ctx, sms, d, m, bound, p, bf, ctx->status, stream, bb_out, side, winners, order);
}

}  // namespace

size_t closure_workspace_bytes(int32_t m, int64_t bound, uint32_t flags) {
  size_t mp = align_up(size_t(m), kB);
  size_t nb = mp / kB;
  return align_up(mp * mp * (use_s16(bound, flags) ? 2 : 4), 256) + align_up(prog_words(nb) * 4, 256) +
         6 * align_up(size_t(m) * 4, 256) + 4096;
}

size_t closure_control_words(int32_t m) {
  return prog_words((size_t(m) + kB - 1) / kB) + size_t(m) + 1;
}

bool closure_small(int32_t m, int64_t bound, uint32_t flags) {
  return m <= (use_s16(bound, flags) ? kClusterMaxWarm<int16_t> : kClusterMaxWarm<int32_t>);
}

int closure_launch(schulze_ctx* ctx, const int32_t* d, int32_t m, int64_t bound, int32_t* p, uint32_t flags,
                   void* ws, cudaStream_t stream, int32_t* beaten_by, int32_t* hint,
                   const int32_t* hint_valid, bool side, int32_t* winners, int32_t* order, uint32_t* control) {
  const bool margin = (flags & SCHULZE_F_MARGIN) != 0;
  if (use_s16(bound, flags))
    return run_closure<int16_t>(ctx, d, m, bound, p, ws, stream, beaten_by, hint, hint_valid, margin, side, winners,
                                order, control);
  return run_closure<int32_t>(ctx, d, m, bound, p, ws, stream, beaten_by, hint, hint_valid, margin, side, winners,
                                order, control);
}

// ------------------------------------------------- allocation-free variant
//
// schulze_strongest_paths_static runs the same kernels as closure_launch on
// scratch that lives in a file-scope device array instead of a context's
// cudaMalloc'ed workspace, for callers that cannot allocate device memory.
// The array is sized for m <= kStaticMaxM; every GPU that loads the library
// holds it until the process exits.

namespace {

constexpr int32_t kStaticMaxM = 1024;
constexpr size_t kStaticMp = 1024;  // kStaticMaxM rounded up to the tile size
constexpr size_t kStaticNb = kStaticMp / kB;
// byte offsets inside the array (each 256-aligned)
constexpr size_t kStW = 0;                                            // W: up to kStaticMp^2 int32
constexpr size_t kStProg = kStW + kStaticMp * kStaticMp * 4;          // progress words + head + abort
constexpr size_t kStRowflag = kStProg + align_up(prog_words(kStaticNb) * 4, 256);
constexpr size_t kStPerm = kStRowflag + kStaticMaxM * 4;
constexpr size_t kStInv = kStPerm + kStaticMaxM * 4;
constexpr size_t kStWarm = kStInv + kStaticMaxM * 4;
constexpr size_t kStCounters = kStWarm + 256;                         // 3 x u64, never read back
constexpr size_t kStaticBytes = kStCounters + 256;

static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
unsigned char* g_static_ptr[kMaxDevices] = {};

// Device address of g_static_scratch on the current device. In host code the
// symbol's name is only a host-side stand-in, so the address is looked up
// once per device, with that device current, and cached.
int static_scratch(int device, unsigned char** out) {
  if (device < 0 || device >= kMaxDevices) return SCHULZE_EINVAL;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_ptr[device]) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) {
      cudaGetLastError();
      return SCHULZE_ECUDA;
    }
    g_static_ptr[device] = static_cast<unsigned char*>(ptr);
  }
  *out = g_static_ptr[device];
  return SCHULZE_OK;
}

template <typename E>
int run_closure_static(unsigned char* base, int device, const int32_t* d, int32_t m, int64_t bound, int32_t* p,
                       int32_t* status, cudaStream_t stream, bool margin) {
  ClosureBufs bf;
  bf.margin = margin;
  bf.W = base + kStW;
  bf.prog = reinterpret_cast<uint32_t*>(base + kStProg);
  bf.rowflag = reinterpret_cast<int32_t*>(base + kStRowflag);
  bf.perm = reinterpret_cast<int32_t*>(base + kStPerm);
  bf.inv = reinterpret_cast<int32_t*>(base + kStInv);
  bf.warm = reinterpret_cast<int32_t*>(base + kStWarm);
  bf.counters = reinterpret_cast<unsigned long long*>(base + kStCounters);
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1)
    return SCHULZE_ECUDA;
  // the array keeps the previous call's contents: the pipeline resets what
  // must start at zero (progress words, queue head, abort flag, row flags)
  return closure_pipeline<E>(nullptr, sms, d, m, bound, p, bf, status, stream);
}

}  // namespace

}  // namespace schulze

extern "C" int schulze_strongest_paths_static(const int32_t* d, int32_t m, int64_t bound, int32_t* p,
                                              uint32_t flags, int32_t* status, schulze_stream_t stream) {
  using namespace schulze;
  if (!d || !p || d == p || m < 1 || bound < 0) return SCHULZE_EINVAL;
  if ((flags & SCHULZE_F_FORCE_S16) && ((flags & SCHULZE_F_FORCE_S32) || bound > 32767)) return SCHULZE_EINVAL;
  if (m > kStaticMaxM) return SCHULZE_ETOOBIG;
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) return SCHULZE_ECUDA;
  unsigned char* base = nullptr;
  if (int rc = static_scratch(device, &base)) return rc;
  const bool margin = (flags & SCHULZE_F_MARGIN) != 0;
  if (use_s16(bound, flags))
    return run_closure_static<int16_t>(base, device, d, m, bound, p, status, stream, margin);
  return run_closure_static<int32_t>(base, device, d, m, bound, p, status, stream, margin);
}
