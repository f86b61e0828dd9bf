// pa_bits.cuh — the spins in device memory, one bit each, and the 32 x 32 bit
// transpose between their layout and the layout the sweeps work on.
//
// In memory a replica is a row of sw words (spin_words): bit b of word k is site
// 32 k + b, set for spin -1; bits past the last site are 0.  A resampled slot's
// spins are then one short contiguous row of its parent (125 bytes at L = 10),
// where int8 site-major rows cost a byte load per site from N far-apart rows:
// the gather and the store of a sweep's tile moved eight times the bytes in 32
// times the loads and took 14 % of a step's sweep at L = 10, R = 1e6.  Whole runs with
// rows of bits against int8 rows: L = 10, R = 1e6 adaptive 224.7 ms (263.7), L = 12,
// R = 77 777 32.1 ms (39.8), L = 8, two populations of 1e5 97.9 ms (143.2, of which the
// overlap was 28.7), reading 1e5 replicas of L = 10 out 15.7 ms (104).
// The sweeps work on site-major words: bit r of a word is replica r of 32
// consecutive slots at one site.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "pa_internal.h"

namespace pa {

// The row of a lattice of size L: SW words, the first NB of them hold sites.
template <int L>
struct Row {
  static constexpr int N = L * L * L, SW = spin_words(N), NB = (N + 31) / 32;
};

// m[i] bit r <-> m[r] bit i, in place (block transposes of 16, 8, 4, 2 and 1 bits;
// the first two are byte permutes): 256 integer instructions for 1024 bits.
__device__ __forceinline__ void transpose32(uint32_t (&m)[32]) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const uint32_t a = m[k], b = m[k + 16];
    m[k] = __byte_perm(a, b, 0x5410);
    m[k + 16] = __byte_perm(a, b, 0x7632);
  }
#pragma unroll
  for (int g = 0; g < 32; g += 16)
#pragma unroll
    for (int k = g; k < g + 8; ++k) {
      const uint32_t a = m[k], b = m[k + 8];
      m[k] = __byte_perm(a, b, 0x6240);
      m[k + 8] = __byte_perm(a, b, 0x7351);
    }
#pragma unroll
  for (int j = 4; j >= 1; j >>= 1) {
    const uint32_t lo = j == 4 ? 0x0F0F0F0Fu : j == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int g = 0; g < 32; g += 2 * j)
#pragma unroll
      for (int k = g; k < g + j; ++k) {
        const uint32_t a = m[k], b = m[k + j];
        m[k] = (a & lo) | ((b << j) & ~lo);
        m[k + j] = ((a >> j) & lo) | (b & ~lo);
      }
  }
}

// Four spins, the low bits of x, as int8 +1 (0x01) / -1 (0xFF).
__device__ __forceinline__ uint32_t spins_to_bytes(uint32_t x) {
  const uint32_t m = ((x & 15u) * 0x00204081u) & 0x01010101u;
  return m * 0xFEu + 0x01010101u;
}
// The reverse: bit 1 of a byte is the sign.
__device__ __forceinline__ uint32_t bytes_to_spins(uint32_t w) {
  return (((w >> 1) & 0x01010101u) * 0x01020408u) >> 24;
}

}  // namespace pa
