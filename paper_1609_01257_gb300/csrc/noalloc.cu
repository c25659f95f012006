// Batched generation for callers that cannot allocate device memory.
//
// rng_batch_create (batch.cu) allocates its work records, a work counter and
// a CUDA graph with cudaMalloc.  Some callers cannot do that: code inside a
// framework whose memory pool owns the whole device and forbids allocations
// beside it, or latency-bound callers that must not pay for an allocation
// (and the device-wide synchronisation a cudaFree implies) on every call.
// This entry point produces the batched form's output with one launch of
// noalloc_kernel, whose blocks find their tile from the instance table alone.
// Up to 64 instances are kernel parameters; more are uploaded to one
// fixed-size array in device global memory declared at file scope below (52
// bytes per instance).  Every GPU that loads the library holds this array
// until the process exits.
//
// Host code cannot use the array's name as a device address (it names a
// host-side stand-in), so the address is looked up with
// cudaGetSymbolAddress, once per device, the first time the entry point runs
// with that device current, and cached.
#include <cuda_runtime.h>
#include <string.h>

#include <algorithm>
#include <mutex>

#include "internal.h"
#include "prng_math.cuh"

namespace {

constexpr uint64_t kUnit = 2048;  // streams of one work unit, in which the limit is counted
constexpr uint64_t kTile = uint64_t(rngi::kGenBlock) * rngi::kNoallocVpt;
constexpr size_t kInstBytes = size_t(RNG_NOALLOC_MAX_INSTANCES) * sizeof(rngi::BatchInstance);
constexpr size_t kScratchBytes = kInstBytes + size_t(RNG_NOALLOC_MAX_INSTANCES) * sizeof(uint32_t);
constexpr int kMaxDevices = 64;

static_assert(sizeof(rngi::BatchInstance) == 48, "table entry size");
static_assert(RNG_NOALLOC_SCRATCH_BYTES == kScratchBytes, "header and scratch size disagree");

// Scratch: [instance table | first tile of each instance].
__device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Host staging (no host allocation per call either): the instances' order and
// the tables of a call with many.
uint32_t g_order[RNG_NOALLOC_MAX_INSTANCES];
struct HostTable {
  rngi::BatchInstance inst[RNG_NOALLOC_MAX_INSTANCES];
  uint32_t first[RNG_NOALLOC_MAX_INSTANCES];
} g_host;
static_assert(sizeof(HostTable) == kScratchBytes, "one upload");

std::mutex g_mu;  // serialises the host side of calls (staging arrays, address cache)
unsigned char *g_scratch_addr[kMaxDevices];

}  // namespace

extern "C" int rng_batch_generate_noalloc(uint32_t count, const uint64_t *streams,
                                          const uint64_t *iterations, const uint64_t *seeds,
                                          uint64_t *const *outs, void *stream, rng_err **err) {
  if (count == 0 || !streams || !iterations || !seeds || !outs)
    return rngi::fail(err, RNG_EINVAL, "rng_batch_generate_noalloc: empty batch or NULL array");
  if (count > RNG_NOALLOC_MAX_INSTANCES)
    return rngi::fail(err, RNG_EINVAL, "rng_batch_generate_noalloc: %u instances, at most %u", count,
                      RNG_NOALLOC_MAX_INSTANCES);
  uint64_t n_units = 0;
  for (uint32_t k = 0; k < count; ++k) {
    if (streams[k] == 0 || streams[k] > (uint64_t(1) << 32) || iterations[k] == 0 || !outs[k])
      return rngi::fail(err, RNG_EINVAL, "rng_batch_generate_noalloc: instance %u has an invalid size or output", k);
    if (iterations[k] > (~uint64_t(0) / 8) / streams[k])
      return rngi::fail(err, RNG_EINVAL, "rng_batch_generate_noalloc: instance %u output size overflows", k);
    if (reinterpret_cast<uintptr_t>(outs[k]) % 8)
      return rngi::fail(err, RNG_EINVAL, "rng_batch_generate_noalloc: instance %u output not 8-byte aligned", k);
    n_units += (streams[k] + kUnit - 1) / kUnit;
  }
  if (n_units > RNG_NOALLOC_MAX_UNITS)
    return rngi::fail(err, RNG_EINVAL,
                      "rng_batch_generate_noalloc: %llu work units (tiles of %llu streams), at most %u",
                      (unsigned long long)n_units, (unsigned long long)kUnit, RNG_NOALLOC_MAX_UNITS);

  std::lock_guard<std::mutex> lk(g_mu);
  int dev = 0;
  cudaError_t st = cudaGetDevice(&dev);
  if (st != cudaSuccess) return rngi::cuda_fail(err, st, "rng_batch_generate_noalloc: cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices)
    return rngi::fail(err, RNG_EINVAL, "rng_batch_generate_noalloc: device %d out of range", dev);
  if (!g_scratch_addr[dev]) {
    // Set-up for this device (the current one): the array's device address.
    void *p = nullptr;
    st = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (st != cudaSuccess) return rngi::cuda_fail(err, st, "rng_batch_generate_noalloc: cudaGetSymbolAddress");
    g_scratch_addr[dev] = static_cast<unsigned char *>(p);
  }

  // Instances with the most rows first (their tiles take longest), each
  // instance's tiles together; std::sort works in place.
  for (uint32_t k = 0; k < count; ++k) g_order[k] = k;
  std::sort(g_order, g_order + count, [&](uint32_t a, uint32_t b) {
    return iterations[a] != iterations[b] ? iterations[a] > iterations[b] : a < b;
  });
  rngi::NoallocArgs args;
  const bool few = count <= rngi::kNoallocFew;
  rngi::BatchInstance *inst = few ? args.few : g_host.inst;
  uint32_t *first = few ? args.few_first : g_host.first;
  uint32_t tiles = 0;
  for (uint32_t i = 0; i < count; ++i) {
    const uint32_t k = g_order[i];
    rngi::BatchInstance &in = inst[i];
    in.out = outs[k];
    in.state = nullptr;
    in.streams = streams[k];
    in.rows = iterations[k];
    in.key = prng::seed_key(seeds[k]);
    // 8-byte stores also on aligned rows: 1000 instances of 1024 streams x 100
    // rows 125 us, 145 with 16-byte ones; one of 2^20 x 300 356 / 393.
    in.vec = 0;
    in.from_hash = 1;
    in.write_state = 0;
    first[i] = tiles;
    tiles += static_cast<uint32_t>((streams[k] + kTile - 1) / kTile);
  }
  args.count = count;
  args.inst = nullptr;
  args.first = nullptr;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (!few) {
    // From pageable memory these copies return once the source has been read,
    // so the staging arrays can be refilled by the next call.
    unsigned char *base = g_scratch_addr[dev];
    st = cudaMemcpyAsync(base, g_host.inst, count * sizeof(rngi::BatchInstance), cudaMemcpyHostToDevice, s);
    if (st == cudaSuccess)
      st = cudaMemcpyAsync(base + kInstBytes, g_host.first, count * sizeof(uint32_t), cudaMemcpyHostToDevice, s);
    if (st != cudaSuccess) return rngi::cuda_fail(err, st, "rng_batch_generate_noalloc: table upload");
    args.inst = reinterpret_cast<const rngi::BatchInstance *>(base);
    args.first = reinterpret_cast<const uint32_t *>(base + kInstBytes);
  }
  st = rngi::launch_noalloc(args, tiles, s);
  return rngi::cuda_fail(err, st, "rng_batch_generate_noalloc: kernel launch");
}
