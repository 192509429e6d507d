// Counting a < b on two 16-bit lanes at once, for lane values below 2^15:
// with the guard bit (bit 15 of each lane) set in a, the difference
// (a | guard) - b lies in [1, 2^16 - 1] in each lane, so no borrow crosses
// the lanes, and its bit 15 is set exactly when a >= b. Three integer
// instructions per pair of lanes (subtract, shift, and-not, add), against
// about five for a packed compare followed by a packed subtract.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace schulze {

constexpr uint32_t kGuard2 = 0x80008000u;  // bit 15 of both 16-bit lanes

// acc's lanes += [a < b] for each lane; a_guarded = a | kGuard2.
__device__ __forceinline__ uint32_t count_lt2(uint32_t acc, uint32_t a_guarded, uint32_t b) {
  return acc + ((~(a_guarded - b) >> 15) & 0x00010001u);
}

// [a < b] on 32 ballots at once, one bit of two positions at a time from the
// lowest up: lt' = (~a & b) | (~(a ^ b) & lt), one logic instruction.
__device__ __forceinline__ uint32_t plane_lt(uint32_t a, uint32_t b, uint32_t lt) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, 0x8E;" : "=r"(r) : "r"(a), "r"(b), "r"(lt));
  return r;
}

// Bit planes of 32 positions below 2^16: w[v] = position v in the low half,
// position v + 16 in the high half (v < 16); on return bit v of w[b] is bit b
// of position v. A 16 x 16 bit transposition of both halves at once, by
// exchanging blocks of 8, 4, 2 and 1 bits.
__device__ __forceinline__ void transpose_planes(uint32_t (&w)[16]) {
#pragma unroll
  for (int v = 0; v < 8; ++v) {  // byte blocks: a byte permutation each
    const uint32_t x = w[v], y = w[v + 8];
    w[v] = __byte_perm(x, y, 0x6240), w[v + 8] = __byte_perm(x, y, 0x7351);
  }
  auto exchange = [&](auto step, uint32_t mask) {
    constexpr int s = decltype(step)::value;
#pragma unroll
    for (int v = 0; v < 16; ++v) {
      if (v & s) continue;
      const uint32_t t = ((w[v] >> s) ^ w[v + s]) & mask;
      w[v + s] ^= t, w[v] ^= t << s;
    }
  };
  exchange(std::integral_constant<int, 4>{}, 0x0F0F0F0Fu);
  exchange(std::integral_constant<int, 2>{}, 0x33333333u);
  exchange(std::integral_constant<int, 1>{}, 0x55555555u);
}

}  // namespace schulze
