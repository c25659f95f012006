// Device helpers shared by the kernels: the jump-ahead tables over GF(2) and
// the XOR / wrapping-sum reductions of the generate-and-checksum kernels.
#pragma once
#include <stdint.h>

namespace rngi {

// Nibble tables of a 64x64 matrix over GF(2): tab[q][e] = the matrix applied
// to the 4-bit value e at bits 4q .. 4q+3.  The product with a vector is then
// 16 table reads and XORs instead of 64 masked XORs, and each table is 16
// words (128 bytes), so a warp's reads of one table never conflict on the
// shared-memory banks.

// From the matrix's columns (col[j] = image of bit j).  By the whole block.
__device__ __forceinline__ void fill_jump_tables(uint64_t (*tab)[16], const uint64_t *__restrict__ cols) {
  for (int idx = threadIdx.x; idx < 16 * 16; idx += blockDim.x) {
    const int q = idx >> 4, e = idx & 15;
    uint64_t acc = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) acc ^= cols[4 * q + i] & (0ull - static_cast<uint64_t>((e >> i) & 1));
    tab[q][e] = acc;
  }
}

// From the tables in memory that jump_tables_kernel wrote.  By the whole block.
__device__ __forceinline__ void load_jump_tables(uint64_t (*tab)[16], const uint64_t *__restrict__ from) {
  for (int idx = threadIdx.x; idx < 16 * 16; idx += blockDim.x) (&tab[0][0])[idx] = from[idx];
}

__device__ __forceinline__ uint64_t apply_jump_tables(const uint64_t (*tab)[16], uint64_t x) {
  uint64_t acc = 0;
#pragma unroll
  for (int q = 0; q < 16; ++q) acc ^= tab[q][(x >> (4 * q)) & 15];
  return acc;
}

// 64-bit XOR and wrapping sum across a warp with 32-bit reductions: the sum
// is split into two 16-bit low parts (no carry can be lost over 32 lanes)
// and the high word, whose sum only matters modulo 2^32.
__device__ __forceinline__ void warp_xor_sum(uint64_t &x, uint64_t &s) {
  const unsigned full = 0xffffffffu;
  const uint32_t xl = __reduce_xor_sync(full, static_cast<uint32_t>(x));
  const uint32_t xh = __reduce_xor_sync(full, static_cast<uint32_t>(x >> 32));
  const uint32_t lo = static_cast<uint32_t>(s);
  const uint32_t a = __reduce_add_sync(full, lo & 0xffffu);
  const uint32_t b = __reduce_add_sync(full, lo >> 16);
  const uint32_t c = __reduce_add_sync(full, static_cast<uint32_t>(s >> 32));
  x = (static_cast<uint64_t>(xh) << 32) | xl;
  s = static_cast<uint64_t>(a) + (static_cast<uint64_t>(b) << 16) + (static_cast<uint64_t>(c) << 32);
}

// XOR of `x` over the block's BLOCK threads, returned to every thread.
// `scratch`: BLOCK / 32 shared words, which the next call may reuse at once.
template <int BLOCK>
__device__ __forceinline__ uint64_t block_xor(uint64_t x, uint64_t *scratch) {
  const unsigned full = 0xffffffffu;
  const uint32_t xl = __reduce_xor_sync(full, static_cast<uint32_t>(x));
  const uint32_t xh = __reduce_xor_sync(full, static_cast<uint32_t>(x >> 32));
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = (static_cast<uint64_t>(xh) << 32) | xl;
  __syncthreads();
  uint64_t r = 0;
#pragma unroll
  for (int w = 0; w < BLOCK / 32; ++w) r ^= scratch[w];
  __syncthreads();
  return r;
}

}  // namespace rngi
