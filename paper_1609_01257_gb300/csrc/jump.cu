// Jump-ahead over GF(2): the update s -> M s is linear, so k iterations are
// M^k.  M's characteristic polynomial p has degree 64 and is irreducible, so
// M^k = c(M) with c = x^k mod p, 64 bits that a few carry-less products give;
// the matrix is then a XOR of the M^i (i < 64) that c names.
//
//  - rng_skip: matrix on the host (a few microseconds), product by a kernel;
//  - banded launches: one kernel computes the tables of all bands, each block
//    its own power, so that neither the host nor a copy is in the way of a
//    generator's first banded launch (they were 64x64 products on the host and
//    an upload).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "internal.h"
#include "prng_math.cuh"
#include "reduce_jump.cuh"

namespace rngi {
namespace {

// a * b modulo x^64 + low.
PRNG_HD uint64_t poly_mul(uint64_t a, uint64_t b, uint64_t low) {
  uint64_t r = 0;
  for (int i = 63; i >= 0; --i) {
    r = (r << 1) ^ (low & (0ull - (r >> 63)));
    r ^= a & (0ull - ((b >> i) & 1));
  }
  return r;
}

// c(M) v: the XOR of M^i v over the bits i of c.
PRNG_HD uint64_t poly_apply(uint64_t c, uint64_t v) {
  uint64_t acc = 0;
  for (; c; c >>= 1) {
    acc ^= v & (0ull - (c & 1));
    v = prng::xorshift_update(v);
  }
  return acc;
}

struct Powers {
  uint64_t low;          // p = x^64 + low
  uint64_t square[64];   // x^(2^i) mod p
  uint64_t col[64][64];  // col[i]: columns of M^i
};

// Built once per process.  M^i e (i < 64) are a basis for any e other than 0
// since p is irreducible, and the coordinates of M^64 e in it are p's low part.
const Powers &powers() {
  static const Powers pw = [] {
    Powers w{};
    uint64_t basis[64] = {}, made_of[64] = {};  // by leading bit: a vector and the M^i e it is the XOR of
    uint64_t v = 1;
    for (int i = 0; i <= 64; ++i, v = prng::xorshift_update(v)) {
      uint64_t r = v, m = i < 64 ? uint64_t(1) << i : 0;
      while (r) {
        const int b = 63 - __builtin_clzll(r);
        if (!basis[b]) {
          basis[b] = r;
          made_of[b] = m;
          break;
        }
        r ^= basis[b];
        m ^= made_of[b];
      }
      if (i == 64) w.low = m;
    }
    w.square[0] = 2;
    for (int i = 1; i < 64; ++i) w.square[i] = poly_mul(w.square[i - 1], w.square[i - 1], w.low);
    for (int j = 0; j < 64; ++j) {
      uint64_t c = uint64_t(1) << j;
      for (int i = 0; i < 64; ++i, c = prng::xorshift_update(c)) w.col[i][j] = c;
    }
    return w;
  }();
  return pw;
}

// x^k mod p.
uint64_t poly_power(uint64_t k) {
  const Powers &w = powers();
  uint64_t c = 1;
  for (int i = 0; k; ++i, k >>= 1)
    if (k & 1) c = poly_mul(c, w.square[i], w.low);
  return c;
}

// Block b: the nibble tables of M^(b * R), given x^R.
__global__ void __launch_bounds__(256) jump_tables_kernel(uint64_t *__restrict__ tables, uint64_t step, uint64_t low) {
  uint64_t c = 1, sq = step;
  for (uint32_t b = blockIdx.x; b; b >>= 1) {
    if (b & 1) c = poly_mul(c, sq, low);
    sq = poly_mul(sq, sq, low);
  }
  const int q = threadIdx.x >> 4, e = threadIdx.x & 15;
  tables[static_cast<uint64_t>(blockIdx.x) * kJumpTableWords + threadIdx.x] =
      poly_apply(c, static_cast<uint64_t>(e) << (4 * q));
}

struct JumpMatrix {
  uint64_t col[64];
};

// Every state is multiplied by the matrix, through nibble tables that each
// block fills from the parameter.  Bound by shared-memory reads: 16 lookups
// of 8 bytes are 32 cycles of an SM's 128 bytes for 32 states (2.3e11
// states/s).  For few states, where jump_wide_kernel's tables cost more.
__global__ void __launch_bounds__(256) jump_kernel(uint64_t *__restrict__ state, uint64_t n, uint64_t id_base,
                                                   uint32_t key, int from_hash, const __grid_constant__ JumpMatrix m) {
  __shared__ uint64_t tab[16][16];
  fill_jump_tables(tab, m.col);
  __syncthreads();
  for (uint64_t s = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; s < n;
       s += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
    const uint64_t v = from_hash ? prng::initial_state(id_base + s, key) : state[s];
    state[s] = apply_jump_tables(tab, v);
  }
}

// The same product with nine lookups: per 32-bit word three tables of 8 bits,
// one of 7, and the last bit of both words together in one of 2.  Entries are
// 8 bytes in 16 copies, one per pair of banks; lane l reads copy l mod 16, so
// that no two lanes of a half warp conflict whatever they look up (one copy
// would conflict about three-fold and be slower than nibbles).  The 1796 x 128
// bytes take an SM's shared memory: one block of 1024 threads per SM.  18
// cycles of shared-memory reads for 32 states instead of 32; 2^26 streams 197
// us (5.4 TB/s of states read and written) against 300 with nibbles.
constexpr int kWideThreads = 1024;
constexpr int kWideEntries = 6 * 256 + 2 * 128 + 4;
constexpr int kWideBytes = kWideEntries * 128;
__host__ __device__ constexpr int kWideEight(int f) { return f * 256; }          // f = 0 .. 5: word f / 3, bits 8 (f % 3) ..
__host__ __device__ constexpr int kWideSeven(int w) { return 1536 + w * 128; }   // word w, bits 24 .. 30
constexpr int kWideLast = 1792;                              // bit 31 and, above it, bit 63

__device__ __forceinline__ uint64_t wide_lookup(const char *lane, uint32_t scaled, int entry) {
  return *reinterpret_cast<const uint64_t *>(lane + scaled + entry * 128);
}

// `lane`: the shared tables plus 8 * (lane mod 16).  Entry e is 128 e bytes on.
__device__ __forceinline__ uint64_t apply_wide(const char *lane, uint64_t x) {
  const uint32_t lo = static_cast<uint32_t>(x), hi = static_cast<uint32_t>(x >> 32);
  uint64_t a = wide_lookup(lane, (lo << 7) & 0x7f80, kWideEight(0));
  uint64_t b = wide_lookup(lane, (lo >> 1) & 0x7f80, kWideEight(1));
  a ^= wide_lookup(lane, (lo >> 9) & 0x7f80, kWideEight(2));
  b ^= wide_lookup(lane, (lo >> 17) & 0x3f80, kWideSeven(0));
  a ^= wide_lookup(lane, (hi << 7) & 0x7f80, kWideEight(3));
  b ^= wide_lookup(lane, (hi >> 1) & 0x7f80, kWideEight(4));
  a ^= wide_lookup(lane, (hi >> 9) & 0x7f80, kWideEight(5));
  b ^= wide_lookup(lane, (hi >> 17) & 0x3f80, kWideSeven(1));
  a ^= wide_lookup(lane, ((lo >> 31) << 7) | ((hi >> 31) << 8), kWideLast);
  return a ^ b;
}

__global__ void __launch_bounds__(kWideThreads, 1) jump_wide_kernel(uint64_t *__restrict__ state, uint64_t n,
                                                                    uint64_t id_base, uint32_t key, int from_hash,
                                                                    const __grid_constant__ JumpMatrix m) {
  extern __shared__ __align__(128) char wide[];
  __shared__ uint64_t nib[16][16];
  fill_jump_tables(nib, m.col);
  __syncthreads();
  // Sixteen threads per entry, one per copy: the stores of a warp fill two
  // entries, 256 contiguous bytes.
  for (int i = threadIdx.x; i < kWideEntries * 16; i += kWideThreads) {
    const int e = i >> 4;
    uint64_t v;
    if (e < 1536) {
      const int f = e >> 8, q = 8 * (f / 3) + 2 * (f % 3);
      v = nib[q][e & 15] ^ nib[q + 1][(e >> 4) & 15];
    } else if (e < kWideLast) {
      const int q = 8 * ((e - 1536) >> 7) + 6;
      v = nib[q][e & 15] ^ nib[q + 1][(e >> 4) & 7];
    } else {
      v = nib[7][(e & 1) << 3] ^ nib[15][((e >> 1) & 1) << 3];
    }
    *reinterpret_cast<uint64_t *>(wide + 8 * static_cast<size_t>(i)) = v;
  }
  __syncthreads();
  const char *lane = wide + 8 * (threadIdx.x & 15);
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * kWideThreads;
  uint64_t s = blockIdx.x * static_cast<uint64_t>(kWideThreads) + threadIdx.x;
  if (from_hash) {
    for (; s < n; s += stride) state[s] = apply_wide(lane, prng::initial_state(id_base + s, key));
    return;
  }
  // The next U states are loaded while U are looked up.
  constexpr int U = 4;
  uint64_t v[U], next[U];
#pragma unroll
  for (int u = 0; u < U; ++u) next[u] = s + u * stride < n ? state[s + u * stride] : 0;
  while (s < n) {
    const uint64_t at = s;
    s += U * stride;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      v[u] = next[u];
      next[u] = s + u * stride < n ? state[s + u * stride] : 0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint64_t r = apply_wide(lane, v[u]);
      if (at + u * stride < n) state[at + u * stride] = r;
    }
  }
}

}  // namespace

cudaError_t launch_jump_tables(uint64_t *tables, uint64_t band_rows, uint32_t count, cudaStream_t st) {
  uint64_t step = poly_power(band_rows), low = powers().low;
  void *params[] = {&tables, &step, &low};
  const cudaError_t e = cudaLaunchKernel(reinterpret_cast<const void *>(&jump_tables_kernel), dim3(count),
                                         dim3(kJumpTableWords), params, 0, st);
  if (e == cudaSuccess) count_launch();
  return e;
}

void jump_matrix(uint64_t k, uint64_t *cols) {
  const Powers &w = powers();
  std::fill(cols, cols + 64, uint64_t(0));
  uint64_t c = poly_power(k);
  for (int i = 0; c; ++i, c >>= 1)
    if (c & 1)
      for (int j = 0; j < 64; ++j) cols[j] ^= w.col[i][j];
}

cudaError_t launch_jump(uint64_t *state, uint64_t n, uint64_t id_base, uint32_t key, int from_hash,
                        const uint64_t *cols, cudaStream_t st) {
  JumpMatrix m;
  std::copy(cols, cols + 64, m.col);
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t sms = static_cast<uint64_t>(device_sm_count(dev));
  void *params[] = {&state, &n, &id_base, &key, &from_hash, &m};
  cudaError_t e;
  if (n >= kJumpWideStreams) {
    const void *fn = reinterpret_cast<const void *>(&jump_wide_kernel);
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kWideBytes);
    if (e == cudaSuccess)
      e = cudaLaunchKernel(fn, dim3(static_cast<unsigned>(sms)), dim3(kWideThreads), params, kWideBytes, st);
  } else {
    const uint64_t blocks_needed = (n + 255) / 256, cap = sms * 8;
    const unsigned grid = static_cast<unsigned>(blocks_needed < cap ? blocks_needed : cap);
    e = cudaLaunchKernel(reinterpret_cast<const void *>(&jump_kernel), dim3(grid ? grid : 1), dim3(256), params, 0, st);
  }
  if (e == cudaSuccess) count_launch();
  return e;
}

}  // namespace rngi
