// Batched elections: thousands of independent elections of uneven size
// (m <= 1024) run in ONE persistent launch. Each CTA takes whole elections
// from a queue ordered by decreasing cost (longest first), and runs the path
// of Sect. 2.1 for each: ballot checks, pairwise tally, winning-votes
// weights, widest-path closure (blocked Floyd-Warshall in the (max, min)
// semiring with four 128-thread tile groups), winners and ranking.
//
// The plan (schulze_batch_create) computes the layout and the job order on
// the host, uploads the job table and reserves per-CTA scratch, so a run
// allocates nothing and can be captured in a CUDA graph.
#include <string.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <numeric>
#include <string>
#include <vector>

#include "count.cuh"
#include "internal.cuh"
#include "tiles.cuh"

namespace schulze {
namespace {

constexpr int kBT = 512;                        // threads per batch CTA
constexpr int kGroups = kBT / tiles::kThreads;  // tile groups of 128 threads
constexpr int32_t kBatchMaxM = 1024;

struct Job {
  int32_t n, m, k, e;
  int64_t ranks_off, mat_off, vec_off;
  int32_t chunk;  // ballots read per tally step (the schedule of the election's m-bucket)
  int32_t gpt;    // tile groups that share the rows of one tally tile (1, 2 or 4)
  int32_t seg;    // schulze_batch_run_host: the segment whose arrival mark the job waits for
  int32_t pad;
};

// Elections are grouped by m into buckets, each with its own tally schedule
// (ballots staged per step, tile groups per tally tile), which
// schulze_batch_autotune times and caches.
constexpr int kBuckets = 5;
constexpr int32_t kBucketMax[kBuckets] = {64, 128, 256, 512, 1024};
inline int bucket_of(int32_t m) {
  int b = 0;
  while (b + 1 < kBuckets && m > kBucketMax[b]) ++b;
  return b;
}
// In the autotuner's cache keys: changed with the kernel, so that choices timed
// on an earlier one (packed compares had no such word) are timed again.
constexpr const char* kTuneKernel = "planes1";
constexpr int kChunkChoices[4] = {8, 16, 32, 64};
constexpr int kGptChoices[3] = {1, 2, 4};
// ballot ids a thread holds for the next step (16: the kernel then fits 128
// registers without spilling, which outweighs the longer steps that 32 allows)
constexpr int kPrefetch = 16;

struct BatchArgs {
  const Job* jobs;
  int32_t njobs;
  uint32_t* head;
  const int32_t* ranks;
  int32_t* d;
  int32_t* p;
  int32_t* winners;
  int32_t* order;
  int32_t* beaten_by;
  unsigned char* scratch;
  size_t slot_bytes;   // per CTA: position planes (the tally), then W over them (the rest), and
  size_t plane_bytes;  // behind these bytes a d slot for when the caller passes no d
  int32_t* status;
  // schulze_batch_run_host: arrival marks of the ballot segments (set by the
  // copy stream after each segment's copy; null otherwise) and the bound on
  // a wait for one, in SM clock cycles
  const int32_t* seg_flag;
  long long wait_limit;
};

// Dynamic shared memory of one batch CTA, reused stage by stage: the tally's
// position rows and its staged planes are carved from `raw`.
constexpr size_t kStageBytes = sizeof(tiles::SmemS32) * kGroups + 2 * tiles::kB * 4;
union BatchSmem {
  unsigned char raw[kStageBytes];
  tiles::SmemS32 t32[kGroups];
  tiles::SmemS16 t16[kGroups];
  int32_t bb[kBatchMaxM];
};

// ------------------------------------------------------------- tally

constexpr int kTT = 64;  // tally tile: 64 x 64 counters per group, 8 x 4 per thread
constexpr int kDiagBlocks = 72;  // 8 x 4 blocks of a diagonal tile on or above the diagonal
constexpr int kPlaneVoters = 32;     // ballots per plane word
constexpr int kPlaneGroups = 256;    // plane groups counted at a time at most (bounds the CTA's scratch; counts fit 16 bits)

__host__ __device__ inline int position_bits(int32_t m, int32_t k) {  // of the largest position (k: unlisted)
  int bits = 0;
  while ((k < m ? k : k - 1) >> bits) ++bits;
  return bits;
}

// Bit planes of the positions on ballots v0 .. v0 + 32 groups - 1 (those past
// n count as all tied): planes[(g * bits + b) * mpad + c] holds bit b of
// candidate c's position on ballots 32 g .. 32 g + 31 (count.cuh: comparing
// two such words bit by bit costs one logic instruction per position bit for
// 32 ballots). Ballots are read `chunk` at a time (the election's schedule),
// their ids two steps ahead in registers, into 16-bit position rows in shared
// memory (unlisted candidates at k), which are turned 32 rows at a time.
// An id out of range or repeated within its ballot sets SCHULZE_EDATA. On full
// rankings a repeated id leaves another candidate out: each row's entries
// carry a bit that alternates between uses of the row, and the turn finds a
// candidate that kept the old one (reading the ids' entries back instead, as
// for shorter ballots, costs as many bank conflicts as writing them: the
// entries of a ballot are 32 random places).
__device__ void make_planes(const Job& jb, const int32_t* __restrict__ ranks, int64_t v0, int32_t groups, int bits,
                            uint32_t* planes, BatchSmem& sm, int32_t* status) {
  const int32_t n = jb.n, m = jb.m, k = jb.k, mpad = int32_t(align_up(size_t(m), kTT));
  const int chunk = jb.chunk, rows = max(chunk, kPlaneVoters);  // chunk * k <= kBT * kPrefetch (plan)
  const int tid = threadIdx.x, lanes = kBT / chunk, vv = tid / lanes, q0 = tid % lanes;
  uint16_t* pos = reinterpret_cast<uint16_t*>(sm.raw);  // [rows][mpad]
  const bool marked = k == m;  // positions below 1024, bit 15 is the mark
  uint32_t mark = 0x8000u;
  if (marked) {
    for (int t = tid; t < rows * mpad / 2; t += kBT) reinterpret_cast<uint32_t*>(pos)[t] = 0u;
    __syncthreads();
  }
  // ids of positions q0 + u * lanes of ballot vv of the step, and of the next
  // one: two sets used in turn (moving one into the other would wait for its loads)
  int32_t ids0[kPrefetch], ids1[kPrefetch];
  auto load_ids = [&](int64_t v, int32_t (&x)[kPrefetch]) {
    const bool have = v + vv < n;
    const int32_t* row = ranks + (v + vv) * k;
#pragma unroll
    for (int u = 0; u < kPrefetch; ++u) {
      const int32_t q = q0 + u * lanes;
      x[u] = (have && q < k) ? __ldcg(row + q) : -1;  // L2 only: see schulze_batch_run_host
    }
  };
  bool bad = false;
  load_ids(v0, ids0);
  load_ids(v0 + chunk, ids1);
  const int64_t vend = v0 + int64_t(groups) * kPlaneVoters;
  int row0 = 0, g0 = 0;  // the step's first row; the plane group of row 0
  auto step = [&](int64_t v, int32_t (&cv)[kPrefetch]) {
    // unlisted candidates, and all of a missing ballot, at position k
    const bool fill = k < m || v + chunk > n;
    if (fill) {
      const uint32_t k2 = (uint32_t(k) | (marked ? mark : 0u)) * 0x10001u;
      const int skip = marked ? int(min(int64_t(chunk), max(int64_t(0), n - v))) : 0;  // (full ballots need no filling)
      uint32_t* p2 = reinterpret_cast<uint32_t*>(pos + (row0 + skip) * mpad);
      for (int t = tid; t < (chunk - skip) * mpad / 2; t += kBT) p2[t] = k2;
      __syncthreads();
    }
    uint16_t* prow = pos + (row0 + vv) * mpad;
    const bool have = v + vv < n;
#pragma unroll
    for (int u = 0; u < kPrefetch; ++u) {
      const int32_t q = q0 + u * lanes, c = cv[u];
      if (!have || q >= k) break;
      if (c < 0 || c >= m) bad = true;
      else prow[c] = uint16_t(uint32_t(q) | (marked ? mark : 0u));
    }
    if (marked) load_ids(v + 2 * chunk, cv);  // in flight from here on
    __syncthreads();
    if (!marked) {
      // a repeated id keeps only one of its positions: the other one sees it
#pragma unroll
      for (int u = 0; u < kPrefetch; ++u) {
        const int32_t q = q0 + u * lanes, c = cv[u];
        if (!have || q >= k) break;
        if (c >= 0 && c < m && prow[c] != uint16_t(q)) bad = true;
      }
      load_ids(v + 2 * chunk, cv);
    }
    row0 += chunk;
    if (row0 < rows) return;
    for (int t = tid; t < rows / kPlaneVoters * mpad; t += kBT) {
      const int gl = t / mpad, c = t - gl * mpad;
      const uint16_t* at = pos + gl * kPlaneVoters * mpad + c;
      uint32_t w[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) w[q] = uint32_t(at[q * mpad]) | (uint32_t(at[(q + 16) * mpad]) << 16);
      transpose_planes(w);
      // (a missing ballot's row was filled with the mark)
      if (marked && c < m && w[15] != (mark ? 0xFFFFFFFFu : 0u) && g0 + gl < groups) bad = true;
      if (g0 + gl < groups) {
        uint32_t* out = planes + int64_t(g0 + gl) * bits * mpad + c;
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (q < bits) out[q * mpad] = w[q];
      }
    }
    __syncthreads();  // the rows are free
    mark ^= 0x8000u, row0 = 0, g0 += rows / kPlaneVoters;
  };
  for (int64_t v = v0; v < vend; v += 2 * chunk) {
    step(v, ids0);
    if (v + chunk < vend) step(v + chunk, ids1);
  }
  if (bad) set_status(status, SCHULZE_EDATA);
}

// counts of one plane group into a thread's RPT x 4 block (rows R0.., columns
// C0..; two 16-bit counters per word)
template <int RPT>
__device__ __forceinline__ void count_group(const uint32_t* S, int bits, int32_t mpad, int32_t R0, int32_t C0,
                                            uint32_t (&acc)[8][2]) {
  uint32_t lt[RPT][4];
#pragma unroll
  for (int r = 0; r < RPT; ++r) lt[r][0] = lt[r][1] = lt[r][2] = lt[r][3] = 0u;
#pragma unroll 2
  for (int b = 0; b < bits; ++b) {
    const uint32_t* P = S + b * mpad;
    uint32_t a[RPT];
    if (RPT == 2) {
      const uint2 x = *reinterpret_cast<const uint2*>(P + R0);
      a[0] = x.x, a[1] = x.y;
    } else {
#pragma unroll
      for (int r = 0; r < RPT; r += 4) {
        const uint4 x = *reinterpret_cast<const uint4*>(P + R0 + r);
        a[r] = x.x, a[r + 1] = x.y, a[r + 2] = x.z, a[r + 3] = x.w;
      }
    }
    const uint4 y = *reinterpret_cast<const uint4*>(P + C0);
    const uint32_t w[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int r = 0; r < RPT; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) lt[r][c] = plane_lt(a[r], w[c], lt[r][c]);
  }
#pragma unroll
  for (int r = 0; r < RPT; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c)
      acc[r][c] += uint32_t(__popc(lt[r][2 * c])) + (uint32_t(__popc(lt[r][2 * c + 1])) << 16);
}

// The counts of `groups` plane groups (at most kPlaneGroups), stored into d
// or (!first) added to it. The four 128-thread groups take 64 x 64 tiles of
// d, two each per round (the planes are read once per round), with jb.gpt
// groups per tile, which then share its rows (and so does a last round with
// one or two tiles left, whatever jb.gpt is). Planes are copied with cp.async
// while the groups before are counted. Full rankings count only the
// tiles above the diagonal and the thread blocks of the diagonal tiles on or
// above it (whole diagonal tiles when groups share tiles), and the last pass
// writes the mirror images d[j][i] = n - d[i][j] with them, eight consecutive
// entries of four rows per thread. Bound by the integer ALU: 4096 elections
// (m to 512, n to 5000) 13.2 ms a CTA, where the logic, counts and adds alone
// take 8.3; the planes before it 5.0, the closure 7.0, the other stages 3.7.
// Counting packed 16-bit compares in the same kernel, the batch took 85.9 ms.
__device__ void count_planes(const Job& jb, const uint32_t* planes, int32_t groups, int bits, bool first, bool last,
                             int32_t* __restrict__ dm, BatchSmem& sm) {
  const int32_t m = jb.m, mpad = int32_t(align_up(size_t(m), kTT)), nbt = mpad / kTT;
  const bool full = jb.k >= m - 1;
  const int tid = threadIdx.x, g = tid / tiles::kThreads, lt = tid % tiles::kThreads;
  const int tx = lt % (kTT / 4), ty = lt / (kTT / 4);
  // Full rankings with one group per tile: the tiles above the diagonal are
  // tasks of their own, and the 8 x 4 thread blocks of the diagonal tiles on
  // or above the diagonal (tx >= 2 ty: 72 of 128 per tile) are packed into
  // tasks of 128 blocks; the blocks below are mirrored with the lower tiles.
  const bool packdiag = full && jb.gpt == 1;
  const int32_t noff = nbt * (nbt - 1) / 2;
  const int32_t ntiles = !full ? nbt * nbt : packdiag ? noff + (nbt * kDiagBlocks + 127) / 128 : nbt * (nbt + 1) / 2;
  const int32_t gwords = bits * mpad;  // words of one plane group
  // two stages of U plane groups each: one barrier per U groups, between which
  // the warps drift apart, so that one warp's population counts (a quarter of
  // the logic rate, on their own unit) run beside the others' logic
  const int U = max(1, min(8, int(kStageBytes / (8 * size_t(max(gwords, 1))))));
  const int32_t uwords = U * gwords;
  const uint32_t* stage = reinterpret_cast<const uint32_t*>(sm.raw);  // [2][U][gwords]
  const uint32_t sbase = uint32_t(__cvta_generic_to_shared(stage));
  auto issue = [&](int32_t q0, int buf) {
    const uint32_t* src = planes + int64_t(q0) * gwords;
    const uint32_t dst = sbase + uint32_t(buf) * uint32_t(uwords) * 4u;
    const int32_t words = min(U, groups - q0) * gwords;  // (negative past the end)
    for (int t = tid; t < words / 4; t += kBT)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + uint32_t(t) * 16u), "l"(src + 4 * t)
                   : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int tpr = 2 * kGroups / jb.gpt;  // tiles per round
  for (int32_t t0 = 0; t0 < ntiles; t0 += tpr) {
    const int T = min(tpr, ntiles - t0);
    const int gr = max(jb.gpt, T == 1 ? 4 : T == 2 ? 2 : 1), teams = kGroups / gr;  // groups per tile, tiles at a time
    // this thread's blocks of d: rows R0.., columns C0.. (8 / gr rows)
    int32_t R0[2], C0[2];
    bool act[2], mir[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int32_t tt = t0 + g / gr + s * teams;
      R0[s] = C0[s] = 0;
      act[s] = tt < t0 + T, mir[s] = false;
      if (!act[s]) continue;
      if (packdiag && tt >= noff) {  // packed blocks of the diagonal tiles
        const int32_t idx = (tt - noff) * 128 + lt;
        act[s] = idx < nbt * kDiagBlocks;
        const int32_t dt = act[s] ? idx / kDiagBlocks : 0;
        int blk = idx % kDiagBlocks, by = 0;
        while (blk >= kTT / 4 - 2 * by) blk -= kTT / 4 - 2 * by, ++by;  // row group by holds 16 - 2 by blocks
        R0[s] = dt * kTT + by * 8, C0[s] = dt * kTT + (2 * by + blk) * 4;
        mir[s] = last && blk >= 2;  // (the first two blocks of a row group hold both halves)
      } else {
        int32_t bi = 0, bj = 0;
        if (full) {  // tiles bi <= bj in order (bi < bj when the diagonal is packed)
          const int32_t dlt = packdiag ? 1 : 0;
          int32_t rem = tt;
          while (rem >= nbt - bi - dlt) rem -= nbt - bi - dlt, ++bi;
          bj = bi + dlt + rem;
        } else {
          bi = tt / nbt, bj = tt % nbt;
        }
        R0[s] = bi * kTT + ty * 8, C0[s] = bj * kTT + tx * 4;
        mir[s] = last && full && bi != bj;
      }
      R0[s] += (g % gr) * (8 / gr);
    }
    uint32_t acc[2][8][2];
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[0][r][0] = acc[0][r][1] = acc[1][r][0] = acc[1][r][1] = 0u;
    issue(0, 0);
    for (int32_t q0 = 0, buf = 0; q0 < groups; q0 += U, buf ^= 1) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();  // these groups' planes are there, the ones before are counted
      issue(q0 + U, buf ^ 1);
      const int qn = min(U, groups - q0);
      for (int q = 0; q < qn; ++q) {
        const uint32_t* S = stage + buf * uwords + q * gwords;
        if (gr == 1) {
          if (act[0]) count_group<8>(S, bits, mpad, R0[0], C0[0], acc[0]);
          if (act[1]) count_group<8>(S, bits, mpad, R0[1], C0[1], acc[1]);
        } else if (gr == 2) {
          if (act[0]) count_group<4>(S, bits, mpad, R0[0], C0[0], acc[0]);
          if (act[1]) count_group<4>(S, bits, mpad, R0[1], C0[1], acc[1]);
        } else {
          if (act[0]) count_group<2>(S, bits, mpad, R0[0], C0[0], acc[0]);
          if (act[1]) count_group<2>(S, bits, mpad, R0[1], C0[1], acc[1]);
        }
      }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (!act[s]) continue;
      int32_t v[8][4];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int32_t i = R0[s] + r;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int32_t j = C0[s] + c;
          v[r][c] = int32_t((acc[s][r][c >> 1] >> (16 * (c & 1))) & 0xFFFFu);
          if (r >= 8 / gr || i >= m || j >= m) continue;
          int32_t* dst = dm + int64_t(i) * m + j;
          if (!first) v[r][c] += *dst;
          *dst = v[r][c];
        }
      }
      if (!mir[s]) continue;
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const int32_t i = R0[s] + r, j = C0[s] + c;
          if (r < 8 / gr && i < m && j < m) dm[int64_t(j) * m + i] = jb.n - v[r][c];
        }
    }
    __syncthreads();  // the stages are free
  }
}

// The election's d: planes and counts, as many plane groups at a time as the
// scratch holds (kPlaneGroups, 8192 ballots, unless the plan had to do with less
// memory).
__device__ void tally(const Job& jb, const int32_t* __restrict__ ranks, int32_t* __restrict__ dm, uint32_t* planes,
                      size_t plane_bytes, BatchSmem& sm, int32_t* status) {
  const int32_t n = jb.n;
  const int bits = position_bits(jb.m, jb.k);
  const size_t group_bytes = size_t(max(bits, 1)) * align_up(size_t(jb.m), kTT) * 4;
  const int32_t most = int32_t(min(size_t(kPlaneGroups), plane_bytes / group_bytes));  // at least 1: W is larger
  for (int64_t v0 = 0; v0 < n; v0 += int64_t(most) * kPlaneVoters) {
    const int32_t groups = int32_t(min(int64_t(most), (n - v0 + kPlaneVoters - 1) / kPlaneVoters));
    make_planes(jb, ranks, v0, groups, bits, planes, sm, status);
    __syncthreads();  // the planes are written
    count_planes(jb, planes, groups, bits, v0 == 0, v0 + int64_t(most) * kPlaneVoters >= n, dm, sm);
  }
  __syncthreads();
}

// ----------------------------------------------------------- stages

constexpr int kMaxTiles = kBatchMaxM / tiles::kB;  // tile rows of the largest election

// What the stages after the tally share: the relabeling of the candidates by
// strength (row sums of d, strongest first), the bounds of the tiles of W and
// the tiles of a phase of the closure that need their update.
struct Shared {
  uint16_t perm[kBatchMaxM], inv[kBatchMaxM];  // new -> old, old -> new
  float key[kBatchMaxM];
  int32_t tmax[kMaxTiles * kMaxTiles], tmin[kMaxTiles * kMaxTiles];
  uint16_t list[kMaxTiles * kMaxTiles];
  alignas(16) int32_t rowbuf[2][tiles::kB];  // the diagonal tile's pivot rows
  int32_t count;
};

// Strongest first, by row sums of d (ties by id): like candidates then share
// tiles and most tile updates can be skipped (see closure.cu).
__device__ void relabel(const int32_t* __restrict__ dm, int32_t m, Shared& sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int32_t i = wid; i < m; i += kBT / 32) {
    float s = 0.f;
    for (int32_t j = lane; j < m; j += 32) s += float(dm[int64_t(i) * m + j]);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if (lane == 0) sh.key[i] = s;
  }
  __syncthreads();
  for (int32_t i = threadIdx.x; i < m; i += kBT) {
    const float mine = sh.key[i];
    int32_t r = 0;
    for (int32_t j = 0; j < m; ++j) r += sh.key[j] > mine || (sh.key[j] == mine && j < i);
    sh.perm[r] = uint16_t(i), sh.inv[i] = uint16_t(r);
  }
  __syncthreads();
}

// W = the weights in strength order, a warp per row, and the tiles' bounds
template <typename E>
__device__ void pack(const Job& jb, const int32_t* __restrict__ dm, int32_t mp, E* __restrict__ W, Shared& sh) {
  const int32_t m = jb.m, n = jb.n, nb = mp / tiles::kB;
  const bool full = jb.k >= m - 1 && n > 0;  // then d[j][i] = n - d[i][j]
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int t = threadIdx.x; t < nb * nb; t += kBT) sh.tmax[t] = 0, sh.tmin[t] = INT32_MAX;
  __syncthreads();
  for (int32_t a = wid; a < mp; a += kBT / 32) {
    const int32_t i = a < m ? sh.perm[a] : -1;
    for (int32_t b = lane; b < mp; b += 32) {
      int32_t out = 0;
      if (i >= 0 && b < m && a != b) {
        const int32_t j = sh.perm[b], x = dm[int64_t(i) * m + j], y = full ? n - x : dm[int64_t(j) * m + i];
        if (x > y) out = x;
      }
      W[int64_t(a) * mp + b] = E(out);
      const int32_t mx = __reduce_max_sync(0xFFFFFFFFu, out);
      const int32_t mn = __reduce_min_sync(0xFFFFFFFFu, i >= 0 && b < m && a != b ? out : INT32_MAX);
      if (lane == 0) {
        const int t = (a / tiles::kB) * nb + b / tiles::kB;
        atomicMax(&sh.tmax[t], mx), atomicMin(&sh.tmin[t], mn);
      }
    }
  }
  __syncthreads();
}

template <typename E>
__device__ void closure(E* W, int32_t m, int32_t mp, BatchSmem& sm, Shared& sh) {
  using Ops = tiles::Ops<E>;
  using tiles::Bounds;
  using tiles::kB;
  const int32_t nb = mp / kB;
  const int g = threadIdx.x / tiles::kThreads, lt = threadIdx.x % tiles::kThreads;
  const tiles::GroupBarrier bar{1 + g};
  auto& ts = sizeof(E) == 2 ? reinterpret_cast<typename Ops::Smem*>(sm.t16)[g]
                            : reinterpret_cast<typename Ops::Smem*>(sm.t32)[g];
  // the group's part of tile t's bounds after its update (reset before it)
  auto bounds = [&](int t, const Bounds& bd) {
    const int32_t mx = __reduce_max_sync(0xFFFFFFFFu, bd.mx), mn = __reduce_min_sync(0xFFFFFFFFu, bd.mn);
    if ((lt & 31) == 0) atomicMax(&sh.tmax[t], mx), atomicMin(&sh.tmin[t], mn);
  };
  // tiles with min(max A, max B) <= min X cannot change; the others of the
  // phase's `total`, at(t) = tile row * nb + tile column, go to sh.list
  auto select = [&](int32_t r, int32_t total, auto at) {
    if (threadIdx.x == 0) sh.count = 0;
    __syncthreads();
    for (int32_t t = threadIdx.x; t < total; t += kBT) {
      const int32_t x = at(t), i = x / nb, j = x % nb;
      if (min(sh.tmax[i * nb + r], sh.tmax[r * nb + j]) > sh.tmin[x]) sh.list[atomicAdd(&sh.count, 1)] = uint16_t(x);
    }
    __syncthreads();
  };
  auto update = [&](int32_t r) {
    for (int32_t t = g; t < sh.count; t += kGroups) {
      const int32_t x = sh.list[t], i = x / nb, j = x % nb, vr = m - i * kB, vc = m - j * kB;
      Ops::load_a(W + int64_t(i) * kB * mp + int64_t(r) * kB, mp, ts, lt);
      Ops::load_b(W + int64_t(r) * kB * mp + int64_t(j) * kB, mp, ts, lt);
      if (lt == 0) sh.tmax[x] = 0, sh.tmin[x] = INT32_MAX;  // (this group's alone until the phase ends)
      Bounds bd;
      Ops::template multiply<true>(W + int64_t(i) * kB * mp + int64_t(j) * kB, mp, ts, lt, bar, bd,
                                   i == j || vr < kB || vc < kB, i == j, vr, vc);
      bounds(x, bd);
      bar.sync();  // the operands are free
    }
    __syncthreads();
  };
  for (int32_t r = 0; r < nb; ++r) {
    const bool close = sh.tmax[r * nb + r] > 0;  // a zero diagonal tile is closed
    __syncthreads();                             // (read by all before its bounds are reset)
    if (g == 0 && close) {
      if (lt == 0) sh.tmax[r * nb + r] = 0, sh.tmin[r * nb + r] = INT32_MAX;
      Bounds bd;
      tiles::diag_closure_local<E>(W, mp, r, m - r * kB, m - r * kB, sh.rowbuf, lt, bar, bd);
      bounds(r * nb + r, bd);
    }
    __syncthreads();
    select(r, 2 * (nb - 1), [&](int32_t t) {  // row, then column panel tiles
      const int32_t v = t < nb - 1 ? t : t - (nb - 1), x = v + (v >= r);
      return t < nb - 1 ? r * nb + x : x * nb + r;
    });
    update(r);
    select(r, (nb - 1) * (nb - 1), [&](int32_t t) {
      const int32_t i = t / (nb - 1), j = t % (nb - 1);
      return (i + (i >= r)) * nb + j + (j >= r);
    });
    update(r);
  }
}

template <typename E>
__device__ void extract(const Job& jb, const E* __restrict__ W, int32_t mp, const BatchArgs& a, BatchSmem& sm,
                        const Shared& sh) {
  const int32_t m = jb.m;
  int32_t* bb = sm.bb;
  for (int32_t i = threadIdx.x; i < m; i += kBT) bb[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int32_t i = w; i < m; i += kBT / 32) {
    int32_t beaten_i = 0;
    for (int32_t j0 = i + 1 + lane; j0 < m; j0 += 32 * 4) {
      int32_t wij[4], wji[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {  // loads first: the transposed ones are strided
        const int32_t j = j0 + 32 * u;
        wij[u] = j < m ? int32_t(W[int64_t(i) * mp + j]) : 0;
        wji[u] = j < m ? int32_t(W[int64_t(j) * mp + i]) : 0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (wji[u] > wij[u]) ++beaten_i;
        else if (wij[u] > wji[u]) atomicAdd(&bb[j0 + 32 * u], 1);
      }
    }
    for (int o = 16; o; o >>= 1) beaten_i += __shfl_xor_sync(0xFFFFFFFFu, beaten_i, o);
    if (lane == 0 && beaten_i) atomicAdd(&bb[i], beaten_i);
  }
  __syncthreads();
  for (int32_t i = threadIdx.x; i < m; i += kBT) {  // relabeled index i, candidate sh.perm[i]
    const int32_t mine = bb[i], id = sh.perm[i];
    if (a.winners) a.winners[jb.vec_off + id] = mine == 0;
    if (a.beaten_by) a.beaten_by[jb.vec_off + id] = mine;
    if (a.order) {
      int32_t pos = 0;
      for (int32_t j = 0; j < m; ++j) {
        const int32_t o = bb[j];
        pos += (o < mine) || (o == mine && sh.perm[j] < id);
      }
      a.order[jb.vec_off + pos] = id;
    }
  }
  if (a.p) {
    int32_t* pm = a.p + jb.mat_off;
    for (int64_t t = threadIdx.x; t < int64_t(m) * m; t += kBT) {
      const int32_t i = int32_t(t / m), j = int32_t(t % m);
      pm[t] = (i == j) ? 0 : int32_t(W[int64_t(sh.inv[i]) * mp + sh.inv[j]]);
    }
  }
  __syncthreads();
}

template <typename E>
__global__ void __launch_bounds__(kBT, 1) batch_kernel(BatchArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BatchSmem& sm = *reinterpret_cast<BatchSmem*>(smem_raw);
  __shared__ int32_t s_job;
  __shared__ Shared sh;
  unsigned char* slot = a.scratch + size_t(blockIdx.x) * a.slot_bytes;
  E* W = reinterpret_cast<E*>(slot);
  uint32_t* planes = reinterpret_cast<uint32_t*>(slot);  // done with before W is packed
  int32_t* dslot = reinterpret_cast<int32_t*>(slot + a.plane_bytes);
  for (;;) {
    if (threadIdx.x == 0) s_job = int32_t(atomicAdd(a.head, 1u));
    __syncthreads();
    const int32_t ji = s_job;
    __syncthreads();
    if (ji >= a.njobs) return;
    const Job jb = a.jobs[ji];
    if (a.seg_flag) {
      // the job's ballots may still be on their way: thread 0 waits (bounded)
      // for its segment's arrival mark, which the copy stream writes after
      // the segment's copy; the ballots are then read from L2, where the copy
      // landed (the tally reads them with L2-only loads, so no line cached in
      // L1 before the mark can be stale)
      __shared__ int32_t s_arrived;
      if (threadIdx.x == 0) {
        const long long t0 = clock64();
        int32_t seen = 0;
        for (;;) {
          asm volatile("ld.acquire.sys.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.seg_flag + jb.seg) : "memory");
          if (seen || clock64() - t0 > a.wait_limit) break;
          __nanosleep(200);
        }
        if (!seen) set_status(a.status, SCHULZE_ETIMEOUT);
        s_arrived = seen;
      }
      __syncthreads();
      if (!s_arrived) return;  // this CTA stops; the status word reports the timeout
    }
    const int32_t* ranks = a.ranks + jb.ranks_off;
    int32_t* dm = a.d ? a.d + jb.mat_off : dslot;
    const int32_t m = jb.m;
    if (jb.n == 0 || jb.k == 0) {
      for (int64_t t = threadIdx.x; t < int64_t(m) * m; t += kBT) dm[t] = 0;
      __syncthreads();
    } else {
      tally(jb, ranks, dm, planes, a.plane_bytes, sm, a.status);
    }
    const int32_t mp = int32_t(align_up(size_t(m), tiles::kB));
    relabel(dm, m, sh);
    pack<E>(jb, dm, mp, W, sh);
    closure<E>(W, m, mp, sm, sh);
    extract<E>(jb, W, mp, a, sm, sh);
  }
}

}  // namespace
}  // namespace schulze

struct schulze_batch {
  schulze_ctx* ctx = nullptr;
  int32_t E = 0;
  bool s16 = true;
  int32_t m_max = 0;
  std::vector<schulze::Job> jobs_host;  // in queue order
  std::vector<int64_t> ranks_off, mat_off, vec_off;  // in the caller's order
  int64_t ranks_elems = 0, mat_elems = 0, vec_elems = 0;
  schulze::Job* jobs_dev = nullptr;
  uint32_t* head = nullptr;
  unsigned char* scratch = nullptr;
  size_t slot_bytes = 0, plane_bytes = 0;
  int grid = 0;
  int32_t tally_policy = 0;  // 0: each m-bucket's ballots per step; 1: eight everywhere
  int32_t order_policy = 0;  // 0 longest first, 1 the caller's order
  int32_t bucket_chunk[schulze::kBuckets] = {32, 32, 32, 16, 16};
  int32_t bucket_gpt[schulze::kBuckets] = {1, 1, 1, 1, 1};
  size_t smem = 0;
  // schulze_batch_run_host (allocated at its first call): device ballots and
  // outputs, the caller's elections cut into segments of about equal ballot
  // bytes with each segment's job table (longest first), the copy stream and
  // one event per segment
  int32_t* host_ranks = nullptr;
  int32_t* host_out = nullptr;  // winners [vec_elems], then order [vec_elems]
  int32_t* seg_flag = nullptr;  // arrival mark per segment
  int32_t* host_one = nullptr;  // page-locked 1, copied into a mark
  schulze::Job* seg_jobs_dev = nullptr;
  std::vector<int32_t> seg_elec0;  // per segment: its first election
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t flags_clear = nullptr;
};

namespace schulze {
namespace {

double job_cost(const Job& j) {
  const double m = j.m, n = j.n, k = j.k;
  const double tally = (k >= m - 1 ? 0.5 : 1.0) * n * m * m;
  const double mp = std::ceil(m / 64.0) * 64.0;
  return tally + 1.5 * mp * mp * mp;
}

// Whether `chunk` ballots of an election with m candidates can be staged: a
// power of two (the CTA's threads divide evenly over the ballots of a step, and
// steps fill whole groups of kPlaneVoters rows or the other way round), the
// position rows (16-bit, at least kPlaneVoters of them) fit the shared
// memory, and a thread holds at most kPrefetch ids of a step (chunk * m <=
// kBT * kPrefetch, as k <= m).
bool chunk_fits(int32_t m, int32_t chunk) {
  const size_t mpad = align_up(size_t(m), kTT);
  return chunk >= 1 && chunk <= kBT && (chunk & (chunk - 1)) == 0 &&
         size_t(std::max(chunk, kPlaneVoters)) * mpad * 2 <= kStageBytes && int64_t(chunk) * m <= int64_t(kBT) * kPrefetch;
}

int32_t job_chunk(const schulze_batch* b, int32_t m) {
  if (b->tally_policy == 1) return 8;
  int32_t c = b->bucket_chunk[bucket_of(m)];
  while (c > 8 && !chunk_fits(m, c)) c /= 2;
  return c;
}

int32_t job_gpt(const schulze_batch* b, int32_t m) { return b->tally_policy == 1 ? 1 : b->bucket_gpt[bucket_of(m)]; }

bool gpt_valid(int32_t g) { return g == 1 || g == 2 || g == 4; }

void order_jobs(schulze_batch* b) {
  std::vector<Job> js(size_t(b->E));
  for (int32_t e = 0; e < b->E; ++e) js[e] = b->jobs_host[e];
  std::sort(js.begin(), js.end(), [](const Job& x, const Job& y) { return x.e < y.e; });
  if (b->order_policy == 0)
    std::stable_sort(js.begin(), js.end(), [](const Job& x, const Job& y) { return job_cost(x) > job_cost(y); });
  for (Job& j : js) j.chunk = job_chunk(b, j.m), j.gpt = job_gpt(b, j.m);
  b->jobs_host = js;
}

int upload_jobs(schulze_batch* b) {
  if (b->E == 0) return SCHULZE_OK;
  if (cudaMemcpy(b->jobs_dev, b->jobs_host.data(), sizeof(Job) * size_t(b->E), cudaMemcpyHostToDevice) !=
      cudaSuccess)
    return SCHULZE_ECUDA;
  return SCHULZE_OK;
}

// One launch over `njobs` jobs of the uploaded table (the whole plan, or a
// subset uploaded by the autotuner), outputs to the per-CTA scratch or the
// caller's buffers.
int launch_jobs(schulze_batch* b, int32_t njobs, const int32_t* ranks, int32_t* d, int32_t* p, int32_t* winners,
                int32_t* order, int32_t* beaten_by, cudaStream_t stream, const Job* jobs = nullptr,
                const int32_t* seg_flag = nullptr) {
  if (cudaMemsetAsync(b->head, 0, 4, stream) != cudaSuccess) return SCHULZE_ECUDA;
  BatchArgs a;
  a.jobs = jobs ? jobs : b->jobs_dev;
  a.seg_flag = seg_flag;
  a.wait_limit = b->ctx->wait_limit_cycles;
  a.njobs = njobs;
  a.head = b->head;
  a.ranks = ranks;
  a.d = d, a.p = p, a.winners = winners, a.order = order, a.beaten_by = beaten_by;
  a.scratch = b->scratch;
  a.slot_bytes = b->slot_bytes;
  a.plane_bytes = b->plane_bytes;
  a.status = b->ctx->status;
  Launch L(b->ctx, stream, "batch_elections", double(njobs));
  if (b->s16)
    batch_kernel<int16_t><<<b->grid, kBT, b->smem, stream>>>(a);
  else
    batch_kernel<int32_t><<<b->grid, kBT, b->smem, stream>>>(a);
  return check_launch();
}

size_t batch_smem(bool s16) {
  (void)s16;
  return sizeof(BatchSmem);
}

}  // namespace
}  // namespace schulze

using namespace schulze;

extern "C" {

int schulze_batch_create(schulze_ctx* ctx, int32_t E, const int32_t* n, const int32_t* m, const int32_t* k,
                         schulze_batch** out) {
  AbiRange abi_range("schulze_batch_create");
  if (!ctx || !out || E < 0 || (E > 0 && (!n || !m || !k))) return SCHULZE_EINVAL;
  *out = nullptr;
  for (int32_t e = 0; e < E; ++e)
    if (m[e] < 1 || m[e] > kBatchMaxM || n[e] < 0 || k[e] < 0 || k[e] > m[e]) return SCHULZE_EINVAL;
  if (cudaSetDevice(ctx->device) != cudaSuccess) return SCHULZE_ECUDA;
  schulze_batch* b = new (std::nothrow) schulze_batch();
  if (!b) return SCHULZE_ENOMEM;
  b->ctx = ctx;
  b->E = E;
  b->ranks_off.resize(size_t(E));
  b->mat_off.resize(size_t(E));
  b->vec_off.resize(size_t(E));
  b->jobs_host.resize(size_t(E));
  int64_t ro = 0, mo = 0, vo = 0;
  for (int32_t e = 0; e < E; ++e) {
    b->ranks_off[e] = ro, b->mat_off[e] = mo, b->vec_off[e] = vo;
    b->jobs_host[e] = Job{n[e], m[e], k[e], e, ro, mo, vo};
    ro += int64_t(n[e]) * k[e];
    mo += int64_t(m[e]) * m[e];
    vo += m[e];
    b->m_max = std::max(b->m_max, m[e]);
    if (n[e] > 32767) b->s16 = false;
  }
  b->ranks_elems = ro, b->mat_elems = mo, b->vec_elems = vo;
  order_jobs(b);
  b->smem = batch_smem(b->s16);
  int per_sm = 0;
  const void* fn = b->s16 ? reinterpret_cast<const void*>(batch_kernel<int16_t>)
                          : reinterpret_cast<const void*>(batch_kernel<int32_t>);
  raise_smem(ctx, fn);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBT, b->smem) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    delete b;
    return SCHULZE_ECUDA;
  }
  b->grid = int(std::max<int64_t>(1, std::min<int64_t>(int64_t(per_sm) * ctx->sm_count, std::max(E, 1))));
  const size_t mp = align_up(size_t(std::max(b->m_max, 1)), tiles::kB);
  const size_t w_bytes = align_up(mp * mp * (b->s16 ? 2 : 4), 256);
  const size_t d_bytes = align_up(size_t(b->m_max) * size_t(b->m_max) * 4, 256);
  size_t plane_words = 0;  // of the largest election's plane groups counted at a time
  for (int32_t e = 0; e < E; ++e) {
    const size_t groups = std::min<size_t>(kPlaneGroups, (size_t(n[e]) + kPlaneVoters - 1) / kPlaneVoters);
    if (k[e] > 0) plane_words = std::max(plane_words, groups * position_bits(m[e], k[e]) * align_up(size_t(m[e]), kTT));
  }
  // planes over W, with room for every plane group of a pass (m = 1024: 10 MB
  // a CTA against W's 2 or 4); where that is not to be had, in W's room alone,
  // in more passes (it holds 5 groups at m = 64 and 51 at m = 1024)
  auto slots = [&](size_t planes) {
    b->plane_bytes = std::max(w_bytes, planes);
    b->slot_bytes = b->plane_bytes + d_bytes;
    const bool ok = cudaMalloc(&b->scratch, b->slot_bytes * size_t(b->grid)) == cudaSuccess;
    if (!ok) cudaGetLastError(), b->scratch = nullptr;
    return ok;
  };
  if (cudaMalloc(&b->jobs_dev, sizeof(Job) * size_t(std::max(E, 1))) != cudaSuccess ||
      cudaMalloc(&b->head, 256) != cudaSuccess || !(slots(align_up(plane_words * 4, 256)) || slots(0))) {
    cudaGetLastError();
    if (b->jobs_dev) cudaFree(b->jobs_dev);
    if (b->head) cudaFree(b->head);
    delete b;
    return SCHULZE_ENOMEM;
  }
  if (int rc = upload_jobs(b)) {
    schulze_batch_destroy(b);
    return rc;
  }
  *out = b;
  return SCHULZE_OK;
}

int schulze_batch_destroy(schulze_batch* b) {
  if (!b) return SCHULZE_EINVAL;
  cudaSetDevice(b->ctx->device);
  cudaDeviceSynchronize();
  cudaFree(b->jobs_dev);
  cudaFree(b->head);
  cudaFree(b->scratch);
  if (b->host_ranks) cudaFree(b->host_ranks);
  if (b->host_out) cudaFree(b->host_out);
  if (b->seg_jobs_dev) cudaFree(b->seg_jobs_dev);
  if (b->seg_flag) cudaFree(b->seg_flag);
  if (b->host_one) cudaFreeHost(b->host_one);
  if (b->copy_stream) cudaStreamDestroy(b->copy_stream);
  if (b->flags_clear) cudaEventDestroy(b->flags_clear);
  delete b;
  return SCHULZE_OK;
}

namespace {

// schulze_batch_run_host's state: at the first call the buffers and the
// segments of the caller's elections (contiguous ballots, about equal ballot
// bytes); at every call the job table: segment after segment, each one's
// elections longest first, with the plan's schedule of that moment.
int host_path_setup(schulze_batch* b) {
  if (!b->host_out) {
    constexpr int kSegments = 8;
    const int nseg = std::max(1, std::min<int>(kSegments, b->E));
    b->seg_elec0.assign(1, 0);
    const double per = double(std::max<int64_t>(b->ranks_elems, 1)) / nseg;
    for (int32_t e = 1; e < b->E && int(b->seg_elec0.size()) < nseg; ++e)
      if (double(b->ranks_off[e]) >= per * double(b->seg_elec0.size())) b->seg_elec0.push_back(e);
    b->seg_elec0.push_back(b->E);
    const size_t ns = b->seg_elec0.size() - 1;
    if (cudaMalloc(&b->host_ranks, sizeof(int32_t) * size_t(std::max<int64_t>(b->ranks_elems, 1))) != cudaSuccess ||
        cudaMalloc(&b->host_out, sizeof(int32_t) * 2 * size_t(std::max<int64_t>(b->vec_elems, 1))) != cudaSuccess ||
        cudaMalloc(&b->seg_jobs_dev, sizeof(Job) * size_t(b->E)) != cudaSuccess ||
        cudaMalloc(&b->seg_flag, sizeof(int32_t) * ns) != cudaSuccess ||
        cudaMallocHost(&b->host_one, sizeof(int32_t)) != cudaSuccess ||
        cudaStreamCreateWithFlags(&b->copy_stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->flags_clear, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      return SCHULZE_ENOMEM;  // what was allocated is freed by schulze_batch_destroy
    }
    *b->host_one = 1;
  }
  std::vector<Job> by_e(size_t(b->E));
  for (const Job& j : b->jobs_host) by_e[size_t(j.e)] = j;
  std::vector<Job> table;
  table.reserve(size_t(b->E));
  for (size_t s = 0; s + 1 < b->seg_elec0.size(); ++s) {
    const size_t t0 = table.size();
    for (int32_t e = b->seg_elec0[s]; e < b->seg_elec0[s + 1]; ++e) {
      table.push_back(by_e[size_t(e)]);
      table.back().seg = int32_t(s);
    }
    std::stable_sort(table.begin() + int64_t(t0), table.end(),
                     [](const Job& x, const Job& y) { return job_cost(x) > job_cost(y); });
  }
  return cudaMemcpy(b->seg_jobs_dev, table.data(), sizeof(Job) * table.size(), cudaMemcpyHostToDevice) == cudaSuccess
             ? SCHULZE_OK
             : SCHULZE_ECUDA;
}

}  // namespace

int schulze_batch_run_host(schulze_batch* b, const int32_t* ranks_host, int32_t* winners_host, int32_t* order_host,
                           schulze_stream_t stream) {
  AbiRange abi_range("schulze_batch_run_host");
  if (!b || (b->ranks_elems > 0 && !ranks_host)) return SCHULZE_EINVAL;
  if (cudaSetDevice(b->ctx->device) != cudaSuccess) return SCHULZE_ECUDA;
  if (b->E == 0) return SCHULZE_OK;
  if (int rc = host_path_setup(b)) return rc;
  const size_t ns = b->seg_elec0.size() - 1;
  int32_t* win = b->host_out;
  int32_t* ord = b->host_out + b->vec_elems;
  // the arrival marks cleared on stream, and the copy stream after that:
  // each segment's ballots, then its mark; meanwhile one launch over every
  // election on stream, each CTA waiting for the mark of its job's segment
  if (cudaMemsetAsync(b->seg_flag, 0, sizeof(int32_t) * ns, stream) != cudaSuccess ||
      cudaEventRecord(b->flags_clear, stream) != cudaSuccess ||
      cudaStreamWaitEvent(b->copy_stream, b->flags_clear, 0) != cudaSuccess)
    return SCHULZE_ECUDA;
  for (size_t s = 0; s < ns; ++s) {
    const int64_t r0 = b->ranks_off[b->seg_elec0[s]];
    const int64_t r1 = b->seg_elec0[s + 1] < b->E ? b->ranks_off[b->seg_elec0[s + 1]] : b->ranks_elems;
    if (r1 > r0 && cudaMemcpyAsync(b->host_ranks + r0, ranks_host + r0, sizeof(int32_t) * size_t(r1 - r0),
                                   cudaMemcpyHostToDevice, b->copy_stream) != cudaSuccess)
      return SCHULZE_ECUDA;
    if (cudaMemcpyAsync(b->seg_flag + s, b->host_one, sizeof(int32_t), cudaMemcpyHostToDevice, b->copy_stream) !=
        cudaSuccess)
      return SCHULZE_ECUDA;
  }
  if (int rc = launch_jobs(b, b->E, b->host_ranks, nullptr, nullptr, winners_host ? win : nullptr,
                           order_host ? ord : nullptr, nullptr, stream, b->seg_jobs_dev, b->seg_flag))
    return rc;
  const size_t vb = sizeof(int32_t) * size_t(b->vec_elems);
  if ((winners_host && cudaMemcpyAsync(winners_host, win, vb, cudaMemcpyDeviceToHost, stream) != cudaSuccess) ||
      (order_host && cudaMemcpyAsync(order_host, ord, vb, cudaMemcpyDeviceToHost, stream) != cudaSuccess))
    return SCHULZE_ECUDA;
  if (cudaStreamSynchronize(stream) != cudaSuccess || cudaStreamSynchronize(b->copy_stream) != cudaSuccess)
    return SCHULZE_ECUDA;
  return SCHULZE_OK;
}

int schulze_batch_layout(const schulze_batch* b, int64_t* ranks_elems, int64_t* mat_elems, int64_t* vec_elems,
                         int64_t* ranks_off, int64_t* mat_off, int64_t* vec_off) {
  if (!b) return SCHULZE_EINVAL;
  if (ranks_elems) *ranks_elems = b->ranks_elems;
  if (mat_elems) *mat_elems = b->mat_elems;
  if (vec_elems) *vec_elems = b->vec_elems;
  for (int32_t e = 0; e < b->E; ++e) {
    if (ranks_off) ranks_off[e] = b->ranks_off[e];
    if (mat_off) mat_off[e] = b->mat_off[e];
    if (vec_off) vec_off[e] = b->vec_off[e];
  }
  return SCHULZE_OK;
}

int schulze_batch_run(schulze_batch* b, const int32_t* ranks, int32_t* d, int32_t* p, int32_t* winners,
                      int32_t* order, int32_t* beaten_by, schulze_stream_t stream) {
  AbiRange abi_range("schulze_batch_run");
  if (!b || (b->ranks_elems > 0 && !ranks)) return SCHULZE_EINVAL;
  if (cudaSetDevice(b->ctx->device) != cudaSuccess) return SCHULZE_ECUDA;
  if (b->E == 0) return SCHULZE_OK;
  return launch_jobs(b, b->E, ranks, d, p, winners, order, beaten_by, stream);
}

int schulze_batch_set_schedule(schulze_batch* b, int32_t tally_policy, int32_t order_policy) {
  if (!b || tally_policy < 0 || tally_policy > 1 || order_policy < 0 || order_policy > 1) return SCHULZE_EINVAL;
  if (cudaSetDevice(b->ctx->device) != cudaSuccess) return SCHULZE_ECUDA;
  if (cudaDeviceSynchronize() != cudaSuccess) return SCHULZE_ECUDA;
  b->tally_policy = tally_policy;
  b->order_policy = order_policy;
  order_jobs(b);
  return upload_jobs(b);
}

int schulze_batch_set_bucket_chunk(schulze_batch* b, int32_t bucket, int32_t chunk) {
  if (!b || bucket < 0 || bucket >= kBuckets || !chunk_fits(kBucketMax[bucket], chunk))
    return SCHULZE_EINVAL;
  if (cudaSetDevice(b->ctx->device) != cudaSuccess) return SCHULZE_ECUDA;
  if (cudaDeviceSynchronize() != cudaSuccess) return SCHULZE_ECUDA;
  b->bucket_chunk[bucket] = chunk;
  order_jobs(b);
  return upload_jobs(b);
}

int schulze_batch_set_bucket_tiles(schulze_batch* b, int32_t bucket, int32_t groups_per_tile) {
  if (!b || bucket < 0 || bucket >= kBuckets || !gpt_valid(groups_per_tile)) return SCHULZE_EINVAL;
  if (cudaSetDevice(b->ctx->device) != cudaSuccess) return SCHULZE_ECUDA;
  if (cudaDeviceSynchronize() != cudaSuccess) return SCHULZE_ECUDA;
  b->bucket_gpt[bucket] = groups_per_tile;
  order_jobs(b);
  return upload_jobs(b);
}

int schulze_batch_bucket_tiles(const schulze_batch* b, int32_t* groups_per_tile) {
  if (!b || !groups_per_tile) return SCHULZE_EINVAL;
  for (int q = 0; q < kBuckets; ++q) groups_per_tile[q] = b->bucket_gpt[q];
  return SCHULZE_OK;
}

int schulze_batch_bucket_schedule(const schulze_batch* b, int32_t* bucket_max_m, int32_t* chunks,
                                  int32_t* elections) {
  if (!b) return SCHULZE_EINVAL;
  for (int q = 0; q < kBuckets; ++q) {
    if (bucket_max_m) bucket_max_m[q] = kBucketMax[q];
    if (chunks) chunks[q] = b->bucket_chunk[q];
    if (elections) elections[q] = 0;
  }
  if (elections)
    for (const Job& j : b->jobs_host) ++elections[bucket_of(j.m)];
  return SCHULZE_OK;
}

int schulze_batch_autotune(schulze_batch* b, const int32_t* ranks, const char* cache_path, int32_t* best_tile,
                           int32_t* best_order, schulze_stream_t stream) {
  AbiRange abi_range("schulze_batch_autotune");
  if (!b || (b->ranks_elems > 0 && !ranks)) return SCHULZE_EINVAL;
  if (cudaSetDevice(b->ctx->device) != cudaSuccess) return SCHULZE_ECUDA;
  // cache keys: GPU, kernel, counter width, then per m-bucket its election
  // count and mean ballot count (the tally schedule), per batch its totals
  // (the order)
  cudaDeviceProp prop;
  cudaGetDeviceProperties(&prop, b->ctx->device);
  auto clean = [](char* key) {
    for (char* c = key; *c; ++c)
      if (*c == ' ' || *c == '\t' || *c == '\n') *c = '_';  // the cache line format splits on blanks
  };
  std::vector<std::pair<std::string, int>> cached;
  if (cache_path) {  // line format: <key> <value>
    if (FILE* f = fopen(cache_path, "r")) {
      char line[512];
      while (fgets(line, sizeof(line), f)) {
        char k2[400];
        int v2;
        if (sscanf(line, "%399s %d", k2, &v2) == 2) cached.emplace_back(k2, v2);
      }
      fclose(f);
    }
  }
  auto lookup = [&](const char* key) {
    int v = -1;
    for (const auto& kv : cached)
      if (kv.first == key) v = kv.second;
    return v;
  };
  std::vector<std::pair<std::string, int>> fresh;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  // best of two timed runs after a warm-up
  auto time_jobs = [&](int32_t njobs, float* ms_out) -> int {
    float best = 1e30f;
    for (int rep = 0; rep < 3; ++rep) {
      cudaEventRecord(e0, stream);
      if (int rc = launch_jobs(b, njobs, ranks, nullptr, nullptr, nullptr, nullptr, nullptr, stream)) return rc;
      cudaEventRecord(e1, stream);
      if (cudaEventSynchronize(e1) != cudaSuccess) return SCHULZE_ECUDA;
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (rep > 0) best = std::min(best, ms);
    }
    *ms_out = best;
    return SCHULZE_OK;
  };
  int rc = SCHULZE_OK;
  b->tally_policy = 0;
  for (int q = 0; q < kBuckets && rc == SCHULZE_OK; ++q) {
    std::vector<Job> sub;
    double nsum = 0.0;
    for (const Job& j : b->jobs_host)
      if (bucket_of(j.m) == q) sub.push_back(j), nsum += j.n;
    if (sub.empty()) continue;
    // the cached value is chunk * 8 + groups per tile
    char key[400];
    snprintf(key, sizeof(key), "%.100s|%s|s16=%d|bucket<=%d|chunk_gpt|elections=%zu|mean_n=%lld", prop.name,
             kTuneKernel, b->s16 ? 1 : 0, kBucketMax[q], sub.size(), (long long)(nsum / double(sub.size())));
    clean(key);
    int best_v = lookup(key);
    if (best_v < 0 || !chunk_fits(kBucketMax[q], best_v / 8) || !gpt_valid(best_v % 8)) {
      // time this bucket's elections alone for every staging size that fits
      // and every number of groups per tally tile
      float best = 1e30f;
      best_v = b->bucket_chunk[q] * 8 + b->bucket_gpt[q];
      for (int c : kChunkChoices) {
        if (!chunk_fits(kBucketMax[q], c)) continue;
        for (int g : kGptChoices) {
          for (Job& j : sub) j.chunk = c, j.gpt = g;
          if (cudaMemcpy(b->jobs_dev, sub.data(), sizeof(Job) * sub.size(), cudaMemcpyHostToDevice) !=
              cudaSuccess) {
            rc = SCHULZE_ECUDA;
            break;
          }
          float ms = 0.f;
          if ((rc = time_jobs(int32_t(sub.size()), &ms)) != SCHULZE_OK) break;
          if (ms < best) best = ms, best_v = c * 8 + g;
        }
        if (rc != SCHULZE_OK) break;
      }
      fresh.emplace_back(key, best_v);
    }
    b->bucket_chunk[q] = best_v / 8;
    b->bucket_gpt[q] = best_v % 8;
  }
  int32_t bo = -1;
  if (rc == SCHULZE_OK) {
    char key[400];
    snprintf(key, sizeof(key), "%.100s|%s|s16=%d|order|E=%d|R=%lld|M=%lld|mmax=%d", prop.name, kTuneKernel, b->s16 ? 1 : 0, b->E,
             (long long)b->ranks_elems, (long long)b->mat_elems, b->m_max);
    clean(key);
    bo = lookup(key);
    if (bo < 0 || bo > 1) {
      float best = 1e30f;
      for (int32_t o = 0; o <= 1 && rc == SCHULZE_OK; ++o) {
        b->order_policy = o;
        order_jobs(b);
        if ((rc = upload_jobs(b)) != SCHULZE_OK) break;
        float ms = 0.f;
        if ((rc = time_jobs(b->E, &ms)) != SCHULZE_OK) break;
        if (ms < best) best = ms, bo = o;
      }
      fresh.emplace_back(key, bo);
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  // the plan's job table back in full with the chosen schedule
  b->order_policy = bo >= 0 ? bo : 0;
  order_jobs(b);
  if (int rc2 = upload_jobs(b)) return rc2;
  if (rc != SCHULZE_OK) return rc;
  if (cache_path && !fresh.empty()) {
    if (FILE* f = fopen(cache_path, "a")) {
      for (const auto& kv : fresh) fprintf(f, "%s %d\n", kv.first.c_str(), kv.second);
      fclose(f);
    }
  }
  if (best_tile) *best_tile = 0;  // each m-bucket's own ballots per step
  if (best_order) *best_order = b->order_policy;
  return SCHULZE_OK;
}

}  // extern "C"
