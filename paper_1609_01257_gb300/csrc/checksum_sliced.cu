// Bit-sliced generate-and-checksum kernel.
//
// The row loop of checksum_kernel is bound by the ALU pipe: five XORs and
// three of the five shifts of every 64-bit update run there (8.07 ALU
// operations per value; 97 % of the pipe's rate and 2.29e12 values/s in a loop
// of rows alone, 2.10e12 in the kernel, on GB300).
// Here 32 streams are held as 64 bit planes (plane j: bit j of each stream,
// one 32-bit word), so that the shifts are only other names for the planes
// and the update is 92 three-input XORs for 32 values (2.9 per value).
// The sum of a row needs the population count of every plane; `popc` runs at
// a quarter of the ALU rate, so each thread first adds its two groups of 32
// streams bit by bit (two logic operations per plane) and counts the 64
// planes of the result: one count and one multiply-add or shift-add per
// value, on other pipes than the XORs.  The XOR of a row comes from the
// update's linearity over GF(2): the XOR of the next row is the update of the
// XOR of this one.
//
// Measured (2^22 streams x 1024 rows, GB300): 1549 us, 2.77e12 values/s,
// against 2517 us for the kernel with a reduction and a barrier in every row
// that did this before and 2049 us for the present checksum_kernel.
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"
#include "prng_math.cuh"
#include "reduce_jump.cuh"

namespace rngi {
namespace {

constexpr int kBlock = static_cast<int>(kSlicedBlock);
constexpr int kGroups = 2;        // groups of 32 streams per thread: 128 registers of planes
constexpr int kBatch = 16;        // rows whose partial sums wait in shared memory
constexpr int kChains = 4;        // carry chains of a row's sum (see row_sum_planes)
static_assert(kSlicedTile == uint64_t(kBlock) * kGroups * 32, "streams of one tile");

// One word from global memory to shared memory without a register (cp.async),
// or 0 when !valid (then nothing is read); done after load_async_wait.
__device__ __forceinline__ void load_async(uint64_t *dst, const uint64_t *src, bool valid) {
  const uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(to), "l"(src), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ void load_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Transposes the 32 x 32 bit matrix x[O .. O + 31] (word k, bit b) <-> (word b, bit k).
template <int O>
__device__ __forceinline__ void transpose32(uint32_t (&x)[64]) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const uint32_t a = x[O + k], b = x[O + k + 16];
    x[O + k] = __byte_perm(a, b, 0x5410);
    x[O + k + 16] = __byte_perm(a, b, 0x7632);
  }
#pragma unroll
  for (int k = 0; k < 32; ++k)
    if (!(k & 8)) {
      const uint32_t a = x[O + k], b = x[O + k + 8];
      x[O + k] = __byte_perm(a, b, 0x6240);
      x[O + k + 8] = __byte_perm(a, b, 0x7351);
    }
#pragma unroll
  for (int i = 2; i >= 0; --i) {
    const int j = 1 << i;
    const uint32_t m = i == 2 ? 0x0f0f0f0fu : i == 1 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if (!(k & j)) {
        const uint32_t t = ((x[O + k] >> j) ^ x[O + k + j]) & m;
        x[O + k + j] ^= t;
        x[O + k] ^= t << j;
      }
  }
}

// The update on bit planes.  With t = s ^ (s << 21), u = t ^ (t >> 35) and
// v = u ^ (u << 4), plane by plane: t[j] = s[j] ^ s[j-21]; u[j] = t[j] from
// plane 29 up and t[j] ^ t[j+35] below; v[j] = u[j] ^ u[j-4].  So
//   v[j] = t[j] ^ t[j-4]                   from plane 33 up,
//   v[j] = t[j] ^ t[j-4] ^ t[j+31]         for planes 29-32,
//   v[j] = t[j] ^ t[j-4] ^ v[j+35]         for planes 4-28
//                                          (v[j+35] = t[j+35] ^ t[j+31]),
//   v[j] = t[j] ^ t[j+35]                  for planes 0-3,
// and a t that has one use is written out as its two planes in a three-input
// XOR: 28 planes of t and 64 of v are left.  In place, from the top down.
__device__ __forceinline__ void update_planes(uint32_t (&p)[64]) {
  uint32_t t[64], low[4], mid[4];
#pragma unroll
  for (int j = 21; j < 64; ++j)
    if (j <= 32 || (j >= 37 && ((j - 37) & 7) < 4) || j >= 61) t[j] = p[j] ^ p[j - 21];
  t[60] = p[60] ^ p[39];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    low[i] = p[i] ^ p[35 + i] ^ p[14 + i];
    mid[i] = t[29 + i] ^ t[25 + i] ^ t[60 + i];
  }
#pragma unroll
  for (int j = 63; j >= 33; --j) {
    const bool own = (j >= 37 && ((j - 37) & 7) < 4) || j >= 60;             // t[j] was kept
    const bool below = j - 4 <= 32 || ((j - 4 - 37) & 7) < 4;                // t[j - 4] was kept
    if (own && below) p[j] = t[j] ^ t[j - 4];
    else if (own) p[j] = t[j] ^ p[j - 4] ^ p[j - 25];
    else p[j] = p[j] ^ p[j - 21] ^ t[j - 4];
  }
#pragma unroll
  for (int j = 28; j >= 4; --j) p[j] = (j >= 21 ? t[j] : p[j]) ^ (j - 4 >= 21 ? t[j - 4] : p[j - 4]) ^ p[j + 35];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    p[29 + i] = mid[i];
    p[i] = low[i];
  }
}

// Sum modulo 2^64 of the thread's 64 values.  The two groups are added plane
// by plane; the carries run in kChains chains of 16 planes that are stepped
// together (one chain of 64 dependent carries left the scheduler short of
// work: 2.89e12 values/s against 3.05e12 with four, in a loop of rows alone;
// eight spill), and a
// chain's last carry is counted at the next chain's first plane.  Counts are
// at most 32, so three 32-bit words hold 24 planes each.
__device__ __forceinline__ uint64_t row_sum_planes(const uint32_t (&a)[64], const uint32_t (&b)[64]) {
  constexpr int L = 64 / kChains;
  uint32_t w[3] = {0, 0, 0}, c[kChains];
#pragma unroll
  for (int k = 0; k < kChains; ++k) c[k] = 0;
#pragma unroll
  for (int i = 0; i < L; ++i)
#pragma unroll
    for (int k = 0; k < kChains; ++k) {
      const int j = k * L + i;
      w[j / 24] += static_cast<uint32_t>(__popc(a[j] ^ b[j] ^ c[k])) << (j % 24);
      c[k] = (a[j] & b[j]) | (c[k] & (a[j] | b[j]));
    }
#pragma unroll
  for (int k = 1; k < kChains; ++k) w[k * L / 24] += static_cast<uint32_t>(__popc(c[k - 1])) << (k * L % 24);
  return static_cast<uint64_t>(w[0]) + (static_cast<uint64_t>(w[1]) << 24) + (static_cast<uint64_t>(w[2]) << 48);
}

// Work is the list of (tile of kSlicedTile streams, quantum of band_rows
// rows) pairs, tile by tile; every block takes an equal contiguous run of it
// (one part of a tile, or the end of one tile and the start of the next), so
// that a grid of one wave ends together whatever the number of tiles.  A run
// that starts inside a tile jumps its states ahead to that row over GF(2).
// band_rows == 0: whole tiles, no jump.  Final states (of runs that reach a
// tile's last row) go to state_out, which may be `state` only when no block
// reads the starting states of a tile that another one ends.
__global__ void __launch_bounds__(kBlock, 3) checksum_sliced_kernel(const RowsLaunch a, unsigned long long *row_xor,
                                                                    unsigned long long *row_sum) {
  __shared__ union {
    uint64_t stage[32][kBlock];          // states between memory and the planes
    uint64_t part[kBatch][kBlock + 1];   // partial sums of a batch of rows
  } mem;
  __shared__ uint64_t jtab[16][16];
  uint64_t(&stage)[32][kBlock] = mem.stage;
  uint64_t(&part)[kBatch][kBlock + 1] = mem.part;
  const uint64_t span = a.s_end - a.s_begin;
  const uint64_t n_tiles = (span + kSlicedTile - 1) / kSlicedTile;
  const uint64_t quantum = a.band_rows ? a.band_rows : a.rows;
  const uint64_t nq = (a.rows + quantum - 1) / quantum;
  const uint64_t total = n_tiles * nq;
  uint64_t w = total / gridDim.x * blockIdx.x + total % gridDim.x * blockIdx.x / gridDim.x;
  const uint64_t b1 = blockIdx.x + 1;
  const uint64_t w_end = total / gridDim.x * b1 + total % gridDim.x * b1 / gridDim.x;
  while (w < w_end) {
    const uint64_t tile = w / nq, q0 = w % nq;
    const uint64_t q1 = nq - q0 < w_end - w ? nq : q0 + (w_end - w);
    const uint64_t r0 = q0 * quantum;
    const uint64_t r1 = q1 * quantum < a.rows ? q1 * quantum : a.rows;
    const uint64_t rel0 = tile * kSlicedTile + threadIdx.x;
    if (q0) {
      load_jump_tables(jtab, a.jump + kJumpTableWords * q0);
      __syncthreads();
    }
    // One group at a time: the thread's 32 states go to its own column of
    // shared memory in rolled loops (unrolled, the hash and the jump are
    // thousands of instructions that run once a tile), all loads in flight
    // together, then to registers, where they are transposed.
    uint32_t p[kGroups][64];
    uint64_t x = 0;
#pragma unroll
    for (int g = 0; g < kGroups; ++g) {
      const uint64_t first = rel0 + static_cast<uint64_t>(32 * g) * kBlock;
      if (a.from_hash) {
#pragma unroll 4
        for (int v = 0; v < 32; ++v) {
          const uint64_t rel = first + static_cast<uint64_t>(v) * kBlock;
          // streams past the end stay 0 and add nothing
          stage[v][threadIdx.x] = rel < span ? prng::initial_state(a.id_base + a.s_begin + rel, a.key) : 0;
        }
      } else {
#pragma unroll 4
        for (int v = 0; v < 32; ++v) {
          const uint64_t rel = first + static_cast<uint64_t>(v) * kBlock;
          load_async(&stage[v][threadIdx.x], a.state + a.s_begin + (rel < span ? rel : 0), rel < span);
        }
        load_async_wait();
      }
      if (q0) {
#pragma unroll 2
        for (int v = 0; v < 32; ++v) stage[v][threadIdx.x] = apply_jump_tables(jtab, stage[v][threadIdx.x]);
      }
#pragma unroll
      for (int v = 0; v < 32; ++v) {
        const uint64_t st = stage[v][threadIdx.x];
        x ^= st;
        p[g][v] = static_cast<uint32_t>(st);
        p[g][32 + v] = static_cast<uint32_t>(st >> 32);
      }
      transpose32<0>(p[g]);
      transpose32<32>(p[g]);
    }
    __syncthreads();  // `part` takes the place of `stage`
    x = block_xor<kBlock>(x, &part[0][0]);
    for (uint64_t r = r0; r < r1; r += kBatch) {
      const int m = r1 - r < kBatch ? static_cast<int>(r1 - r) : kBatch;
#pragma unroll 1
      for (int q = 0; q < m; ++q) {
        part[q][threadIdx.x] = row_sum_planes(p[0], p[1]);
#pragma unroll
        for (int g = 0; g < kGroups; ++g) update_planes(p[g]);
      }
      __syncthreads();
      constexpr int kPerRow = kBlock / kBatch;  // threads that add up one row
      const int row = threadIdx.x / kPerRow, k = threadIdx.x % kPerRow;
      uint64_t s = 0;
#pragma unroll
      for (int i = 0; i < kBlock / kPerRow; ++i) s += part[row][k + kPerRow * i];
#pragma unroll
      for (int d = kPerRow / 2; d; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
      if (k == 0 && row < m) atomicAdd(row_sum + r + row, static_cast<unsigned long long>(s));
      if (threadIdx.x == kBlock - 1)
        for (int q = 0; q < m; ++q) {
          atomicXor(row_xor + r + q, static_cast<unsigned long long>(x));
          x = prng::xorshift_update(x);
        }
      __syncthreads();
    }
    if (a.write_state && q1 == nq) {
#pragma unroll
      for (int g = 0; g < kGroups; ++g) {
        transpose32<0>(p[g]);
        transpose32<32>(p[g]);
#pragma unroll
        for (int v = 0; v < 32; ++v)
          stage[v][threadIdx.x] = (static_cast<uint64_t>(p[g][32 + v]) << 32) | p[g][v];
#pragma unroll 4
        for (int v = 0; v < 32; ++v) {
          const uint64_t rel = rel0 + static_cast<uint64_t>(32 * g + v) * kBlock;
          if (rel < span) a.state_out[a.s_begin + rel] = stage[v][threadIdx.x];
        }
      }
    }
    __syncthreads();
    w += q1 - q0;
  }
}

}  // namespace

const void *checksum_sliced_kernel_fn() { return reinterpret_cast<const void *>(&checksum_sliced_kernel); }

}  // namespace rngi
