// (max, min) tile routines shared by the single-election closure and the
// batched elections: the diagonal-tile Floyd-Warshall and the 64 x 64 x 64
// tile update X = max(X, A (x) B). Each runs on a group of 128 threads that
// synchronise through `Bar`: the whole block, or one named barrier per group
// when a block runs several groups side by side.
#pragma once

#include "internal.cuh"

namespace schulze {
namespace tiles {

constexpr int kB = 64;         // block / tile size
constexpr int kThreads = 128;  // threads of one tile group
constexpr int kRM = 8;         // rows per thread in a tile update
constexpr int kRN = 4;         // columns per thread in a tile update
constexpr int kTX = kB / kRN;  // 16 column groups x 8 row groups = 128 threads

// All threads of the block.
struct BlockBarrier {
  __device__ __forceinline__ void sync() const { __syncthreads(); }
};

// Named barrier `id` (1..15) over the 128 threads of one group.
struct GroupBarrier {
  int id;
  __device__ __forceinline__ void sync() const { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }
};

// Smallest and largest entry of a tile (one thread's part of it): mx over
// every entry off the matrix diagonal, mn over those of them in the tile's
// first vr rows and vc columns (rows past the last candidate with edges never
// change and columns past the last candidate do not exist). A tile update
// X = max(X, A (x) B) with min(mx(A), mx(B)) <= mn(X) changes nothing.
struct Bounds {
  int32_t mx, mn;
};

// Closes the diagonal tile (r, r) in place by plain Floyd-Warshall over its
// 64 vertices. Thread t keeps row t / 2, columns 32 (t % 2) .. + 31 in
// registers; at step k the two owners of row k publish it through shared
// memory and p[i][k] comes from the thread itself or its neighbour lane.
// Row k and column k do not change during step k (min(x, y) <= x). The
// tile's diagonal may pick up cycle widths; it never changes an off-diagonal
// entry and is zeroed on output. The caller's barrier has to follow.
// 16-bit lanes stay packed two to a word (two lane updates per min and max).
template <typename E, class Bar>
__device__ void diag_closure_local(E* __restrict__ W, int32_t ld, int32_t r, int32_t vr, int32_t vc,
                                   int32_t (*rowbuf)[kB], int tid, const Bar& bar, Bounds& bd) {
  constexpr int kPer = 4 / int(sizeof(E));  // entries per word
  constexpr int kWords = 32 / kPer;         // words of a thread's half row
  const int i = tid >> 1, half = tid & 1;
  E* base = W + (int64_t(r) * kB + i) * ld + int64_t(r) * kB + half * 32;
  uint32_t v[kWords];
#pragma unroll
  for (int q = 0; q < kWords / 4; ++q) {
    const uint4 x = __ldcg(reinterpret_cast<const uint4*>(base) + q);
    v[4 * q] = x.x, v[4 * q + 1] = x.y, v[4 * q + 2] = x.z, v[4 * q + 3] = x.w;
  }
#pragma unroll
  for (int k = 0; k < kB; ++k) {
    uint32_t* rb = reinterpret_cast<uint32_t*>(rowbuf[k & 1]) + half * kWords;
    if (i == k) {
#pragma unroll
      for (int c = 0; c < kWords; c += 4)
        *reinterpret_cast<uint4*>(&rb[c]) = make_uint4(v[c], v[c + 1], v[c + 2], v[c + 3]);
    }
    bar.sync();
    const int kk = k & 31;
    uint32_t mine = v[kk / kPer];
    if (sizeof(E) == 2) mine = __byte_perm(mine, 0, (kk & 1) ? 0x3232 : 0x1010);
    const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, mine, 1);
    const uint32_t a = ((k >> 5) == half) ? mine : other;  // p[i][k] (in both lanes)
#pragma unroll
    for (int c = 0; c < kWords; c += 4) {
      const uint4 b = *reinterpret_cast<const uint4*>(&rb[c]);
      auto step = [&](uint32_t& x, uint32_t y) {
        if (sizeof(E) == 2) x = __vmaxs2(x, __vmins2(a, y));
        else x = uint32_t(max(int32_t(x), min(int32_t(a), int32_t(y))));
      };
      step(v[c], b.x), step(v[c + 1], b.y), step(v[c + 2], b.z), step(v[c + 3], b.w);
    }
  }
#pragma unroll
  for (int q = 0; q < kWords / 4; ++q)
    __stcg(reinterpret_cast<uint4*>(base) + q, make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
  // this thread's part of the tile's bounds
  bd = Bounds{0, INT32_MAX};
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    const int j = half * 32 + c;
    const int32_t x = sizeof(E) == 2 ? int32_t(int16_t(v[c / kPer] >> (16 * (c & 1)))) : int32_t(v[c / kPer]);
    if (j == i) continue;
    bd.mx = max(bd.mx, x);
    if (i < vr && j < vc) bd.mn = min(bd.mn, x);
  }
}

// Shared-memory operand layouts of one tile update.
struct SmemS32 {
  int32_t A[kB][kB];  // A[k][i] = W(ti, r)[i][k] (transposed)
  int32_t B[kB][kB];  // B[k][j] = W(r, tj)[k][j]
};
struct SmemS16 {
  uint32_t A[kB][kB];  // A[k][i] = W(ti, r)[i][k] in both 16-bit halves
  uint16_t B[kB][kB];  // B[k][j]
};

// Tile update X = max(X, A (x) B) by lane format, in parts: load_a and load_b
// stage the 64 x 64 operands at Ag and Bg (row stride ld), multiply loads X
// from Cg, synchronises through bar (operands staged), computes and stores X.
// The caller synchronises before the operands are staged anew or X is read.
// With kBounds multiply returns this thread's part of the bounds of X (edge:
// X touches the matrix diagonal (diag) or the padding, vr and vc as above).
template <typename E>
struct Ops;

template <>
struct Ops<int32_t> {
  using Smem = SmemS32;
  static __device__ __forceinline__ void load_a(const int32_t* Ag, int32_t ld, Smem& sm, int tid) {
    const int i = tid % kB, k0 = (tid / kB) * 32;  // row i, 32 consecutive k
    const int4* src = reinterpret_cast<const int4*>(Ag + int64_t(i) * ld + k0);
    int4 v[8];  // every load in flight before the first store
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __ldcg(src + q);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      sm.A[k0 + 4 * q + 0][i] = v[q].x;
      sm.A[k0 + 4 * q + 1][i] = v[q].y;
      sm.A[k0 + 4 * q + 2][i] = v[q].z;
      sm.A[k0 + 4 * q + 3][i] = v[q].w;
    }
  }
  static __device__ __forceinline__ void load_b(const int32_t* Bg, int32_t ld, Smem& sm, int tid) {
    const int k0 = tid / 16, c4 = tid % 16;
    int4 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __ldcg(reinterpret_cast<const int4*>(Bg + int64_t(k0 + 8 * q) * ld) + c4);
#pragma unroll
    for (int q = 0; q < 8; ++q) *reinterpret_cast<int4*>(&sm.B[k0 + 8 * q][c4 * 4]) = v[q];
  }
  template <bool kBounds, class Bar>
  static __device__ __forceinline__ void multiply(int32_t* Cg, int32_t ld, Smem& sm, int tid,
                                                  const Bar& bar, Bounds& bd, bool edge = false, bool diag = false,
                                                  int32_t vr = kB, int32_t vc = kB) {
    const int tx = tid % kTX, ty = tid / kTX;
    int32_t acc[kRM][kRN];
#pragma unroll
    for (int rr = 0; rr < kRM; ++rr) {
      int4 v = __ldcg(reinterpret_cast<const int4*>(Cg + int64_t(ty * kRM + rr) * ld + tx * kRN));
      acc[rr][0] = v.x, acc[rr][1] = v.y, acc[rr][2] = v.z, acc[rr][3] = v.w;
    }
    bar.sync();
    // two k-steps per three-input max: max(c, min(a, b), min(a', b'))
#pragma unroll 2
    for (int k = 0; k < kB; k += 2) {
      int32_t a[2][8], bb[2][4];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        int4 a0 = *reinterpret_cast<const int4*>(&sm.A[k + h][ty * kRM]);
        int4 a1 = *reinterpret_cast<const int4*>(&sm.A[k + h][ty * kRM + 4]);
        int4 b = *reinterpret_cast<const int4*>(&sm.B[k + h][tx * kRN]);
        a[h][0] = a0.x, a[h][1] = a0.y, a[h][2] = a0.z, a[h][3] = a0.w;
        a[h][4] = a1.x, a[h][5] = a1.y, a[h][6] = a1.z, a[h][7] = a1.w;
        bb[h][0] = b.x, bb[h][1] = b.y, bb[h][2] = b.z, bb[h][3] = b.w;
      }
#pragma unroll
      for (int rr = 0; rr < kRM; ++rr)
#pragma unroll
        for (int c = 0; c < kRN; ++c)
          acc[rr][c] = __vimax3_s32(acc[rr][c], min(a[0][rr], bb[0][c]), min(a[1][rr], bb[1][c]));
    }
#pragma unroll
    for (int rr = 0; rr < kRM; ++rr)
      __stcg(reinterpret_cast<int4*>(Cg + int64_t(ty * kRM + rr) * ld + tx * kRN),
             make_int4(acc[rr][0], acc[rr][1], acc[rr][2], acc[rr][3]));
    if (!kBounds) return;
    int32_t mx = 0, mn = INT32_MAX;
    if (!edge) {
#pragma unroll
      for (int rr = 0; rr < kRM; ++rr) {
        mx = __vimax3_s32(mx, acc[rr][0], acc[rr][1]), mx = __vimax3_s32(mx, acc[rr][2], acc[rr][3]);
        mn = __vimin3_s32(mn, acc[rr][0], acc[rr][1]), mn = __vimin3_s32(mn, acc[rr][2], acc[rr][3]);
      }
    } else {
#pragma unroll
      for (int rr = 0; rr < kRM; ++rr)
#pragma unroll
        for (int c = 0; c < kRN; ++c) {
          const int i = ty * kRM + rr, j = tx * kRN + c;
          if (diag && i == j) continue;
          mx = max(mx, acc[rr][c]);
          if (i < vr && j < vc) mn = min(mn, acc[rr][c]);
        }
    }
    bd = Bounds{mx, mn};
  }
};

// Two 16-bit lanes per word.
template <>
struct Ops<int16_t> {
  using Smem = SmemS16;
  static __device__ __forceinline__ void load_a(const int16_t* Ag, int32_t ld, Smem& sm, int tid) {
    const int i = tid % kB, k0 = (tid / kB) * 32;
    const uint4* src = reinterpret_cast<const uint4*>(Ag + int64_t(i) * ld + k0);
    uint4 v[4];  // every load in flight before the first store
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = __ldcg(src + q);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t w4[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        uint32_t lo = w4[h] & 0xFFFFu, hi = w4[h] >> 16;
        sm.A[k0 + 8 * q + 2 * h][i] = lo | (lo << 16);
        sm.A[k0 + 8 * q + 2 * h + 1][i] = hi | (hi << 16);
      }
    }
  }
  static __device__ __forceinline__ void load_b(const int16_t* Bg, int32_t ld, Smem& sm, int tid) {
    const int k0 = tid / 8, c8 = tid % 8;
    uint4 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = __ldcg(reinterpret_cast<const uint4*>(Bg + int64_t(k0 + 16 * q) * ld) + c8);
#pragma unroll
    for (int q = 0; q < 4; ++q) *reinterpret_cast<uint4*>(&sm.B[k0 + 16 * q][c8 * 8]) = v[q];
  }
  template <bool kBounds, class Bar>
  static __device__ __forceinline__ void multiply(int16_t* Cg, int32_t ld, Smem& sm, int tid,
                                                  const Bar& bar, Bounds& bd, bool edge = false, bool diag = false,
                                                  int32_t vr = kB, int32_t vc = kB) {
    const int tx = tid % kTX, ty = tid / kTX;
    uint32_t acc[kRM][kRN / 2];
#pragma unroll
    for (int rr = 0; rr < kRM; ++rr) {
      uint2 v = __ldcg(reinterpret_cast<const uint2*>(Cg + int64_t(ty * kRM + rr) * ld + tx * kRN));
      acc[rr][0] = v.x, acc[rr][1] = v.y;
    }
    bar.sync();
#pragma unroll 2
    for (int k = 0; k < kB; k += 2) {
      uint32_t a[2][8], b[2][2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint4 a0 = *reinterpret_cast<const uint4*>(&sm.A[k + h][ty * kRM]);
        uint4 a1 = *reinterpret_cast<const uint4*>(&sm.A[k + h][ty * kRM + 4]);
        uint2 bv = *reinterpret_cast<const uint2*>(&sm.B[k + h][tx * kRN]);
        a[h][0] = a0.x, a[h][1] = a0.y, a[h][2] = a0.z, a[h][3] = a0.w;
        a[h][4] = a1.x, a[h][5] = a1.y, a[h][6] = a1.z, a[h][7] = a1.w;
        b[h][0] = bv.x, b[h][1] = bv.y;
      }
#pragma unroll
      for (int rr = 0; rr < kRM; ++rr)
#pragma unroll
        for (int w = 0; w < 2; ++w)
          acc[rr][w] = __vimax3_s16x2(acc[rr][w], __vmins2(a[0][rr], b[0][w]), __vmins2(a[1][rr], b[1][w]));
    }
#pragma unroll
    for (int rr = 0; rr < kRM; ++rr)
      __stcg(reinterpret_cast<uint2*>(Cg + int64_t(ty * kRM + rr) * ld + tx * kRN), make_uint2(acc[rr][0], acc[rr][1]));
    if (!kBounds) return;
    int32_t mx = 0, mn = INT32_MAX;
    if (!edge) {
      uint32_t mx2 = 0u, mn2 = 0x7FFF7FFFu;
#pragma unroll
      for (int rr = 0; rr < kRM; ++rr) {
        mx2 = __vimax3_s16x2(mx2, acc[rr][0], acc[rr][1]);
        mn2 = __vimin3_s16x2(mn2, acc[rr][0], acc[rr][1]);
      }
      mx = max(int32_t(int16_t(mx2 & 0xFFFFu)), int32_t(int16_t(mx2 >> 16)));
      mn = min(int32_t(int16_t(mn2 & 0xFFFFu)), int32_t(int16_t(mn2 >> 16)));
    } else {
#pragma unroll
      for (int rr = 0; rr < kRM; ++rr)
#pragma unroll
        for (int c = 0; c < kRN; ++c) {
          const int i = ty * kRM + rr, j = tx * kRN + c;
          const int32_t x = int16_t(acc[rr][c >> 1] >> (16 * (c & 1)));
          if (diag && i == j) continue;
          mx = max(mx, x);
          if (i < vr && j < vc) mn = min(mn, x);
        }
    }
    bd = Bounds{mx, mn};
  }
};

// X(ti, tj) = max(X, W(ti, r) (x) W(r, tj)), ending with the barrier that
// frees the shared operands.
template <typename E, class Bar>
__device__ __forceinline__ void tile_update(E* W, int32_t ld, int32_t ti, int32_t tj, int32_t r,
                                            typename Ops<E>::Smem& sm, int tid, const Bar& bar) {
  Ops<E>::load_a(W + int64_t(ti) * kB * ld + int64_t(r) * kB, ld, sm, tid);
  Ops<E>::load_b(W + int64_t(r) * kB * ld + int64_t(tj) * kB, ld, sm, tid);
  Bounds bd;
  Ops<E>::template multiply<false>(W + int64_t(ti) * kB * ld + int64_t(tj) * kB, ld, sm, tid, bar, bd);
  bar.sync();
}

}  // namespace tiles
}  // namespace schulze
