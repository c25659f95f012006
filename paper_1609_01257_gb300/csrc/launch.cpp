// Host-side launch code of the kernels: shape selection (values per thread,
// store width, grid, bands) and the launches themselves, but for the
// jump-ahead's (jump.cu).  The kernels are in kernels.cu and
// checksum_sliced.cu; this file holds no device code.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "internal.h"

namespace rngi {
namespace {

int occupancy(const void *fn, uint32_t block) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, static_cast<int>(block), 0) !=
          cudaSuccess ||
      n < 1)
    n = 1;
  return n;
}


}  // namespace

int device_sm_count(int device) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1)
    sms = 1;
  return sms;
}

// Values per thread for 256-thread blocks, from sweeps of the row kernel on
// GB300 (152 SMs) writing 4-32 GiB per launch with one tile per block:
//  - 24 streams per thread (one 48 KiB run per block and row, one resident
//    block per SM) was fastest from 2^22 to 2^26 streams;
//  - from 2^20 up to that, one stream per thread (thousands of short tiles):
//    7.14-7.23 TB/s at 2^20 and 7.33-7.38 at 2^21 on every GPU tried, where
//    shapes of about 128 tiles (fewer blocks than SMs) ran at 7.4 TB/s on some
//    GPUs but 6.1 on others;
//  - below 2^20 about 128 tiles (one long-running block on most SMs) stayed
//    fastest on average: 8 per thread at 2^18 (6.3-7.6 TB/s against 6.5 for
//    one per thread), 2 at 2^16 (6.2-7.4 against 6.5).
uint32_t default_vpt(uint64_t streams, int sms) {
  const uint64_t M = uint64_t(1) << 20;
  if (streams >= 7 * M / 2) return 24;
  if (streams >= M) return 1;
  (void)sms;
  const uint64_t v = streams / (uint64_t(kGenBlock) * 128);
  for (uint32_t c : {32u, 16u, 8u, 4u, 2u})
    if (v >= c) return c;
  return 1;
}

// Values per thread of the staged row kernel for rows that do not start on
// 128-byte lines (a stream count that is not a multiple of 16), or 0 to keep
// the unstaged kernel.  Measured on GB300 (1024 rows, GB/s): 2^22 + 1
// streams 6968 unstaged (24 per thread) vs 6882 staged at best, so from 3.5 M
// streams the unstaged kernel stays; 3,000,017 streams 4411 unstaged vs 6762
// staged at 8 per thread; 1,000,003 streams 4204 vs 6297 at 2; 250,001
// streams 5642 at 4; 65,537 streams 4976 at 8 (banded).
uint32_t staged_vpt(uint64_t streams, uint32_t requested, int sms) {
  if (requested) return requested == 1 || requested == 2 || requested == 4 || requested == 6 || requested == 8
                            ? requested : 0;
  const uint64_t M = uint64_t(1) << 20;
  if (streams >= 7 * M / 2) return 0;
  if (streams >= 2 * M) return 8;
  if (streams >= M / 2) return 2;
  const uint64_t tiles8 = (streams + uint64_t(kGenBlock) * 8 - 1) / (uint64_t(kGenBlock) * 8);
  return tiles8 * 2 < static_cast<uint64_t>(sms) ? 8 : 4;  // 8 when the launch will be banded
}

// Row buffers of the bulk-copy row kernel for `vpt` values per thread (0 if
// that count has no bulk variant).
uint32_t bulk_buffers(uint32_t vpt) {
  switch (vpt) {
    case 4: return 8;
    case 8: return 12;
    case 10: return 9;
    case 16: return 6;
    case 24: return 4;
    default: return 0;
  }
}

namespace {

// Blocks that write at the same time hold their copies to this rate (bytes a
// second, all together): see Pacer.  With 152 blocks and 2^22 streams x 256
// rows 7.5, 7.6, 7.7 and 7.8e12 gave 7422, 7518, 7621 and 7711 GB/s; a
// copy-only kernel held 7.88e12 and fell back at 8.0e12.  For the whole GB300
// (HBM3e, 7.9 TB/s nominal; fills 7.55 to 7.65 on those measured): on a
// partition, or a part whose memory takes less, the pace does not hold the
// copies back and they run as they did without it.
constexpr double kWriteRate = 7.7e12;

uint32_t pace_of(uint64_t blocks) {
  return static_cast<uint32_t>(static_cast<double>(blocks) / kWriteRate * 1e9 * 1048576.0);
}

uint32_t ceil16(uint64_t v) { return static_cast<uint32_t>((v + 15) / 16 * 16); }

}  // namespace

// The bulk-copy kernels for one launch of `rows` rows over `streams` streams
// when the caller leaves the shape to the library, for rows on 128-byte lines
// (`lined`) and off them; nb == 0: keep the register or staged kernels.
// may_band: the rows may be split into bands; out_rows: rows of the output
// (the ring's, when rows wrap).  One block per SM, all with equal shares:
// tiles and bands come to whole rounds of the SMs, because a paced block does
// not use what another leaves (1000003 streams x 512 rows, 16 values per
// thread: 304 tiles of 3296 in two rounds 7555 GB/s, 245 of 4096 6106).  A
// block's step per row takes about 0.3 us with 8 values per thread and 0.38
// to 0.44 with 16, so tiles are as wide as the threads' values allow.
// Where the lines lie (GB300, us before / with this plan):
//  - up to 4096 streams, the whole row in a block: 300 x 100 44 / 14, 1001 x
//    4096 60 / 18, 4096 x 65536 333 / 294; rows on the lines keep register
//    stores below 256 MB (4096 x 4096 32 / 33) and 16 rows per band, and 4096 x
//    64 off a line (9.9 / 19.8);
//  - 5500 x 1024 74 / 24, 20001 x 16384 549 / 359, 65537 x 255 58 / 35, 131073
//    x 1024 188 / 154; below 128 rows register stores (direct_vpt) are faster;
//  - 250001 x 255 81 / 82 (in bands 82), x 1024 293 / 281: from 1024 rows;
//  - 400001 x 64 51 / 41, 1000003 x 128 167 / 150, 3000017 x 128 453 / 428, 2^22
//    + 1 x 64 317 / 306; below 32 rows even or worse up to 2^21 streams (2^21 x
//    31 off a line 125 staged / 89);
//  - on the lines, 2^20 x 255 307 / 292, 2^22 x 128 602 / 584, 65536 x 4096 293 /
//    294 (and 340 where 128 unpaced SMs are past the ceiling); 2^22 x 64 308 /
//    324, 2^24 x 32 656 / 690 (each tile's loads are exposed);
//  - rings on the lines: what a small one overwrites stays in the L2, 2^20 x
//    512 into 16 or 64 rows 489 or 550 / 580, into 128 (1 GB) 611 / 581;
//  - without bands, fewer tiles than half the SMs would be cut into pieces of a
//    few KB, each of which takes its block the 0.4 us: rings of 65536 x 8192
//    553 / 3400, 70001 x 300 41 / 146.
BulkPlan bulk_plan(uint64_t streams, uint64_t rows, bool lined, bool may_band, uint64_t out_rows, uint32_t sms) {
  constexpr uint64_t M = uint64_t(1) << 20;
  BulkPlan p;
  const bool ring = out_rows < rows;
  const uint64_t bytes = 8 * streams * out_rows;
  uint64_t units;
  if (streams <= 4096) {
    if (!may_band || rows < (lined ? 16 * uint64_t(sms) : streams % 16 == 0 && streams > 1024 ? 128 : 64)) return p;
    if (lined && streams > 1024 && bytes < 256 * M) return p;
    const uint64_t bands = std::min<uint64_t>(sms, rows / 16);
    p.multi = true;
    p.vpt = 1;
    while (streams > uint64_t(kGenBlock) * p.vpt) p.vpt *= 2;
    p.nb = 6;
    p.tile_w = static_cast<uint32_t>(streams);
    p.band_rows = (rows + bands - 1) / bands;
    units = (rows + p.band_rows - 1) / p.band_rows;
  } else {
    const bool many = streams >= 7 * M / 2;
    // One tile of 24 values per thread rather than two half empty ones of 16.
    p.vpt = streams <= uint64_t(kGenBlock) * 24 ? 24 : 16;
    p.nb = bulk_buffers(p.vpt);
    const uint64_t most = uint64_t(kGenBlock) * p.vpt;
    const uint64_t tiles = (streams + most - 1) / most;
    if (!may_band && tiles * 2 <= sms) return BulkPlan{};
    if (lined) {
      if (many ? rows < 128 : rows <= 128 || bytes < (ring || tiles < sms ? 1024 : 256) * M) return BulkPlan{};
    } else if (rows < (streams < uint64_t(sms) * 1024 ? 128 : streams >= 2 * M ? 16 : 32)) {
      return BulkPlan{};
    }
    const bool narrow = tiles < sms && tiles > sms / 4 && rows < 1024 && streams <= uint64_t(sms) * 2048;
    if (rows < 32 || narrow) {
      // Few rows of many streams: one block per tile, so that a tile's last
      // copies and the next one's start overlap (2^22 + 1 x 16 103, register
      // stores 123).  Fewer tiles than SMs, too many for bands that are worth
      // their jumps: the narrowest tiles whose copies are not too small.
      p.vpt = 8;
      p.nb = bulk_buffers(p.vpt);
      p.tile_w = kGenBlock * 8;
      return p;
    }
    uint64_t bands = 1;
    if (tiles >= sms) {
      const uint64_t rounds = (tiles + sms - 1) / sms;
      p.tile_w = ceil16((streams + rounds * sms - 1) / (rounds * sms));
    } else {
      if (may_band) bands = std::max<uint64_t>(1, std::min<uint64_t>(sms / tiles, rows / 16));
      p.tile_w = ceil16((streams + sms / bands - 1) / (sms / bands));
      if (bands > 1) p.band_rows = (rows + bands - 1) / bands;
    }
    // Every value of a thread takes its time in a row, used or not: equal shares
    // that come to at most 10 values run with 10 (622593 x 100 76 us, with 16
    // values 97, staged 85; 330001 x 300 113 / 138).
    if (bands == 1 && p.tile_w <= kGenBlock * 10) {
      p.vpt = 10;
      p.nb = bulk_buffers(p.vpt);
    }
    units = (streams + p.tile_w - 1) / p.tile_w * (bands > 1 ? (rows + p.band_rows - 1) / p.band_rows : 1);
  }
  p.blocks = static_cast<uint32_t>(std::min<uint64_t>(units, sms));
  // Outputs that the 129 MB L2 can take are written as fast as it takes them.
  if (bytes >= 128 * M) p.pace = pace_of(p.blocks);
  return p;
}

// Rows off the lines without a bulk plan (small launches): register stores
// all the same when the staged kernel would have few blocks, each with a
// barrier per row.  GB300, staged / direct us: 65537 x 16 14.3 / 6.5, x 64
// 39 / 12; 20001 x 100 59 / 12; 131073 x 64 39 / 16; 250001 x 16 11.9 / 9.8.
uint32_t direct_vpt(uint64_t streams) {
  if (streams >= 384 * 1024) return 0;
  return streams >= 100 * 1024 ? 4 : streams >= 64 * 1024 ? 2 : 1;
}

LaunchShape rows_shape(uint64_t streams, uint32_t vpt, uint32_t block, int device, uint32_t max_grid,
                       uint32_t width, int policy) {
  LaunchShape sh;
  sh.block = block ? block : kGenBlock;
  const int sms = device_sm_count(device);
  if (policy == kStoreBulk) {
    // Every row written by bulk copies, whatever its alignment.
    sh.vpt = vpt ? vpt : 8;
    sh.bulk_forced = bulk_buffers(sh.vpt) != 0;
    sh.width = 1;
    const uint64_t tiles = (streams + uint64_t(kGenBlock) * sh.vpt - 1) / (uint64_t(kGenBlock) * sh.vpt);
    uint64_t grid = max_grid && max_grid < tiles ? max_grid : tiles;
    if (grid > 0x7fffffffull) grid = 0x7fffffffull;
    sh.grid = sh.bulk_forced && sh.block == kGenBlock ? static_cast<uint32_t>(grid ? grid : 1) : 0;
    return sh;
  }
  sh.bulk_auto = policy == kStoreStreaming && vpt == 0 && sh.block == kGenBlock && max_grid == 0 && width == 0;
  sh.sms = static_cast<uint32_t>(sms);
  if (sh.block == kGenBlock && streams % 16 != 0) {
    const uint32_t v = staged_vpt(streams, vpt, sms);
    if (v) {
      sh.staged = true;
      sh.vpt = v;
      sh.width = 1;
      const uint64_t tiles = (streams + uint64_t(kGenBlock) * v - 1) / (uint64_t(kGenBlock) * v);
      uint64_t grid = max_grid && max_grid < tiles ? max_grid : tiles;
      if (grid > 0x7fffffffull) grid = 0x7fffffffull;
      sh.grid = static_cast<uint32_t>(grid ? grid : 1);
      return sh;
    }
  }
  if (vpt == 0) vpt = sh.block == kGenBlock ? default_vpt(streams, sms) : 8;
  sh.vpt = vpt;
  // One 8-byte store per value measured fastest once a thread holds six or
  // more streams (see the shape sweep in the design notes); below that the
  // widest store the alignment allows.
  sh.width = width ? width : (vpt >= 6 ? 1 : 4);
  // Occupancy of the variant that will run (policy and store width change
  // the register count).
  const void *fn = rows_kernel_fn(vpt, static_cast<int>(sh.width), sh.block == kGenBlock ? policy : kStoreStreaming, sh.block);
  if (!fn) {
    sh.grid = 0;
    return sh;
  }
  const uint64_t tiles = (streams + static_cast<uint64_t>(sh.block) * vpt - 1) /
                         (static_cast<uint64_t>(sh.block) * vpt);
  // One block per tile by default: the hardware hands tiles out in order as
  // blocks finish, which measured ~10% faster than a persistent grid-stride
  // loop (tiles running at the same time stay adjacent in memory).  max_grid
  // asks for fewer blocks; then each block strides over the tiles.
  uint64_t grid = max_grid ? max_grid : tiles;
  if (grid > tiles) grid = tiles;
  if (grid > 0x7fffffffull) grid = 0x7fffffffull;
  sh.grid = static_cast<uint32_t>(grid ? grid : 1);
  return sh;
}

LaunchShape resolve_shape(const LaunchShape &sh, const RowsLaunch &a, bool may_band) {
  LaunchShape r = sh;
  r.bulk = BulkPlan{};
  if (!a.out) return r;
  const uint64_t span = a.s_end - a.s_begin;
  const bool lined = a.pitch % 16 == 0 && reinterpret_cast<uintptr_t>(a.out) % 128 == 0;
  if (sh.bulk_forced) {
    r.bulk.vpt = sh.vpt;
    r.bulk.nb = bulk_buffers(sh.vpt);
    r.bulk.tile_w = kGenBlock * sh.vpt;
  } else if (sh.bulk_auto) {
    r.bulk = bulk_plan(span, a.rows, lined, may_band, a.ring_rows ? std::min(a.ring_rows, a.rows) : a.rows, sh.sms);
  }
  if (!r.bulk.nb) {
    const uint32_t v = sh.bulk_auto && !lined ? direct_vpt(span) : 0;
    if (v) {
      r.direct = true;
      r.staged = false;
      r.vpt = v;
      r.width = 2;
      r.grid = static_cast<uint32_t>((span + uint64_t(kGenBlock) * v - 1) / (uint64_t(kGenBlock) * v));
    }
    return r;
  }
  r.vpt = r.bulk.vpt;
  r.staged = false;
  r.width = 1;
  const uint64_t tiles = (span + r.bulk.tile_w - 1) / r.bulk.tile_w;
  uint64_t grid = tiles;
  if (sh.bulk_forced && sh.grid && sh.grid < tiles) grid = sh.grid;  // a grid the caller asked for
  if (grid > 0x7fffffffull) grid = 0x7fffffffull;
  r.grid = static_cast<uint32_t>(grid ? grid : 1);
  return r;
}

cudaError_t launch_rows(const RowsLaunch &a, const LaunchShape &sh, int store_policy, cudaStream_t st,
                        LaunchInfo *info) {
  if (a.band_rows && (a.ring_rows || !a.jump || (a.write_state && !a.from_hash && a.state_out == a.state)))
    return cudaErrorInvalidValue;
  // Widest store the output's alignment allows: every row must start on an
  // 8*W-byte boundary (pitch a multiple of W, base aligned to 8*W bytes).
  int width = 1;
  const uintptr_t base = reinterpret_cast<uintptr_t>(a.out);
  for (int w : {4, 2})
    if (a.out && a.pitch % w == 0 && base % (8 * w) == 0) {
      width = w;
      break;
    }
  if (width > static_cast<int>(sh.width)) width = static_cast<int>(sh.width);
  // Rows that do not start on 128-byte lines (a pitch that is not a multiple
  // of 16 values, or an output off a line): a warp's run of 8-byte stores
  // then touches nine 32-byte sectors instead of eight.  Shapes chosen for
  // such rows (sh.staged), and shapes of 1-8 values per thread whose output
  // starts off a line, run the staged row kernel, which stores line-aligned
  // pieces; the tiles are the same.
  const uint32_t vpt = sh.vpt;
  const bool small_vpt = vpt == 1 || vpt == 2 || vpt == 4 || vpt == 6 || vpt == 8;
  const bool bulk = a.out && sh.bulk.nb;
  const bool staged = !bulk && !sh.direct && a.out && !a.ring_rows && sh.block == kGenBlock && small_vpt &&
                      (sh.staged || a.pitch % 16 != 0 || base % 128 != 0);
  const int policy = store_policy == kStoreBulk ? kStoreStreaming : store_policy;
  const void *fn = bulk && sh.bulk.multi
                       ? (a.band_rows && a.pitch == a.s_end - a.s_begin ? rows_multi_kernel_fn(vpt, a.out_mode) : nullptr)
                   : bulk   ? (a.ring_rows ? rows_bulk_ring_kernel_fn(vpt, sh.bulk.nb, a.out_mode)
                                           : rows_bulk_kernel_fn(vpt, sh.bulk.nb, a.band_rows != 0, a.out_mode))
                   : staged ? rows_staged_kernel_fn(vpt, a.band_rows != 0, a.out_mode)
                            : rows_kernel_fn(vpt, width, policy, sh.block, a.band_rows != 0, a.out_mode);
  uint64_t grid = sh.grid;
  const uint64_t span = a.s_end - a.s_begin;
  if (!fn) return cudaErrorInvalidValue;
  size_t smem = 0;
  if (bulk) {
    smem = sh.bulk.multi ? rows_multi_smem_bytes() : rows_bulk_smem_bytes(vpt, sh.bulk.nb);
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  RowsLaunch args = a;
  const uint64_t tile_w = bulk ? sh.bulk.tile_w : uint64_t(sh.block) * vpt;
  args.tile_w = static_cast<uint32_t>(tile_w);
  args.pace = bulk ? sh.bulk.pace : 0;
  void *params[] = {&args};
  if (a.band_rows) {
    // One block per (tile, band) unit, unless the shape asked for fewer.
    const uint64_t tiles = (span + tile_w - 1) / tile_w;
    const uint64_t units = tiles * ((a.rows + a.band_rows - 1) / a.band_rows);
    if (grid >= tiles) grid = units < 0x7fffffffull ? units : 0x7fffffffull;
  }
  if (bulk && sh.bulk.blocks && sh.bulk.blocks < grid) grid = sh.bulk.blocks;
  if (grid > 0x7fffffffull) grid = 0x7fffffffull;
  cudaError_t e = cudaLaunchKernel(fn, dim3(static_cast<unsigned>(grid)), dim3(sh.block), params, smem, st);
  if (e == cudaSuccess) {
    count_launch();
    if (info) {
      info->kernel = bulk ? RNG_KERNEL_BULK : staged ? RNG_KERNEL_STAGED : RNG_KERNEL_REGISTER;
      info->vpt = vpt;
      info->block = sh.block;
      info->grid = static_cast<uint32_t>(grid);
      info->row_buffers = bulk ? sh.bulk.nb : 0;
      info->band_rows = a.band_rows;
    }
  }
  return e;
}

cudaError_t launch_init(uint64_t *state, uint64_t n, uint64_t id_base, uint32_t key,
                        cudaStream_t st) {
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t blocks_needed = (n + 255) / 256;
  const uint64_t cap = static_cast<uint64_t>(device_sm_count(dev)) * 8;
  const unsigned grid = static_cast<unsigned>(blocks_needed < cap ? blocks_needed : cap);
  void *params[] = {&state, &n, &id_base, &key};
  cudaError_t e = cudaLaunchKernel(init_kernel_fn(), dim3(grid ? grid : 1), dim3(256), params, 0, st);
  if (e == cudaSuccess) count_launch();
  return e;
}

cudaError_t launch_copy(uint64_t *dst, const uint64_t *src, uint64_t n, cudaStream_t st) {
  int dev = 0;
  cudaGetDevice(&dev);
  // One block per SM keeps enough stores in flight for the host link (1, 2,
  // 4, 8 and 16 blocks per SM measured within 5 % of each other) while the
  // generation kernel of the next chunk runs beside them.
  const uint64_t blocks_needed = (n + 255) / 256;
  const uint64_t cap = static_cast<uint64_t>(device_sm_count(dev));
  const unsigned grid = static_cast<unsigned>(blocks_needed < cap ? blocks_needed : cap);
  void *params[] = {&dst, &src, &n};
  cudaError_t e = cudaLaunchKernel(copy_kernel_fn(), dim3(grid ? grid : 1), dim3(256), params, 0, st);
  if (e == cudaSuccess) count_launch();
  return e;
}

// Register and staged row kernels (bound by HBM writes): bands only when the
// tiles cannot cover half the SMs (128 unbanded tiles of 2^16 streams ran at
// 7.37 TB/s, three bands of them at 6.25: more SMs than HBM takes writes
// from, see Pacer in kernels.cu); then about two (tile, band) units per SM
// (16 tiles of 4096 streams: 19 bands 6.6 TB/s, 10 bands 4.7 TB/s).  A bulk
// plan carries its own bands.
// Checksum kernel (bound by integer issue): bands whenever the tiles leave
// resident block slots empty, up to about four units per slot, so that the
// last wave of units is a small part of the launch.
// Bands hold at least 128 rows (64 in the checksum kernel), which amortises
// each unit's jump.
uint64_t choose_band_rows(uint64_t streams, uint64_t rows, const LaunchShape &sh, int device, bool checksum,
                          uint32_t out) {
  const uint64_t sms = static_cast<uint64_t>(device_sm_count(device));
  const uint64_t tiles = (streams + uint64_t(sh.block) * sh.vpt - 1) / (uint64_t(sh.block) * sh.vpt);
  const uint64_t min_band = checksum ? 64 : 128;
  if (!checksum && sh.bulk.nb && !sh.bulk_forced) return sh.bulk.band_rows;  // part of the plan
  const void *fn = checksum     ? checksum_kernel_fn(sh.vpt, true, out)
                   : sh.bulk.nb ? rows_bulk_kernel_fn(sh.vpt, sh.bulk.nb, true, out)
                   : sh.staged  ? rows_staged_kernel_fn(sh.vpt, true, out)
                                : rows_kernel_fn(sh.vpt, 1, kStoreStreaming, sh.block, true, out);
  if (!fn || rows < 2 * min_band) return 0;  // no banded variant of this shape, or too few rows
  uint64_t target;
  if (checksum) {
    const uint64_t slots = sms * static_cast<uint64_t>(std::max(1, occupancy(fn, sh.block)));
    if (tiles >= slots) return 0;
    target = 4 * slots;
  } else {
    if (tiles * 2 >= sms) return 0;
    target = 2 * sms;
  }
  uint64_t bands = (target + tiles - 1) / tiles;
  if (bands > rows / min_band) bands = rows / min_band;
  if (bands > kMaxBands) bands = kMaxBands;
  if (bands < 2) return 0;
  return (rows + bands - 1) / bands;
}

uint64_t checksum_split_rows(uint64_t streams, uint64_t rows, uint32_t vpt, int device, uint32_t out) {
  if (rows < 2 * 64) return 0;  // before the occupancy query, 0.2 us of the host
  const uint64_t tile = uint64_t(kGenBlock) * vpt, tiles = (streams + tile - 1) / tile;
  const void *fn = checksum_kernel_fn(vpt, true, out);
  if (!fn) return 0;
  const uint64_t slots = static_cast<uint64_t>(device_sm_count(device)) * occupancy(fn, kGenBlock);
  const auto use = [&](uint64_t units) {
    return static_cast<double>(units) / static_cast<double>((units + slots - 1) / slots * slots);
  };
  if (tiles < slots || use(tiles) > 0.93) return 0;
  double best = use(tiles) + 0.02;
  uint64_t band = 0;
  for (uint64_t bands = 2; bands <= 8 && rows / bands >= 64; ++bands) {
    const uint64_t br = (rows + bands - 1) / bands;
    if (use(tiles * ((rows + br - 1) / br)) <= best) continue;
    best = use(tiles * ((rows + br - 1) / br));
    band = br;
  }
  return band;
}

uint32_t checksum_vpt(uint64_t span, uint64_t rows, uint32_t vpt, int device) {
  if (vpt) return vpt;
  const uint64_t sms = static_cast<uint64_t>(device_sm_count(device));
  // Large launches run at the ALU rate with 8 to 32 values per thread; the
  // start of a unit (jump, reductions) weighs least at 16.  Small launches are
  // bound by one block's rows, one after another, so they take fewer values
  // per thread and more blocks (us on GB300 at 4 / 8 / 16: 8192 x 1024 25 / 30
  // / 40; 65536 x 256 32 / 31 / 40; 1000003 x 16 37 / 27 / 29; 262144 x 256
  // 62 / 62 / 60; 65536 x 4096 176 / 167 / 173) unless there are many tiles
  // anyway: many tiles of few rows wait for their atomics on the same few
  // words, so from five tiles of 16 values an SM on the larger ones are taken (8
  // / 16: 2^22 x 15 50 / 43, 6000001 x 8 42 / 35).  A tile that would be mostly past
  // the end of the streams is halved.
  const uint64_t values = span * rows;
  uint32_t v = values >= (uint64_t(1) << 26) || span >= kGenBlock * 16 * 5 * sms ? 16
               : values >= (uint64_t(1) << 24) || span >= kGenBlock * 8 * sms    ? 8
                                                                                 : 4;
  while (v > 1) {
    const uint64_t tile = uint64_t(kGenBlock) * v, tiles = (span + tile - 1) / tile;
    if (span * 5 >= tiles * tile * 4) break;
    if (tiles > 8) break;
    v /= 2;
  }
  return v;
}

cudaError_t launch_checksum(const RowsLaunch &a, uint32_t vpt, uint64_t *row_xor, uint64_t *row_sum,
                            cudaStream_t st, LaunchInfo *info) {
  const uint64_t span = a.s_end - a.s_begin;
  int dev = 0;
  cudaGetDevice(&dev);
  const int sms = device_sm_count(dev);
  if (a.band_rows && (!a.jump || (a.write_state && !a.from_hash && a.state_out == a.state))) return cudaErrorInvalidValue;
  const void *fn = checksum_kernel_fn(vpt, a.band_rows != 0, a.out_mode);
  if (!fn) return cudaErrorInvalidValue;
  const uint64_t tiles = (span + uint64_t(kGenBlock) * vpt - 1) / (uint64_t(kGenBlock) * vpt);
  const uint64_t units = a.band_rows ? tiles * ((a.rows + a.band_rows - 1) / a.band_rows) : tiles;
  const uint64_t resident = uint64_t(sms) * occupancy(fn, kGenBlock);
  const unsigned grid = static_cast<unsigned>(std::max<uint64_t>(1, std::min(units, resident)));
  RowsLaunch args = a;
  unsigned long long *rx = reinterpret_cast<unsigned long long *>(row_xor);
  unsigned long long *rs = reinterpret_cast<unsigned long long *>(row_sum);
  void *params[] = {&args, &rx, &rs};
  cudaError_t e = cudaLaunchKernel(fn, dim3(grid), dim3(kGenBlock), params, 0, st);
  if (e == cudaSuccess) {
    count_launch();
    *info = {RNG_KERNEL_CHECKSUM, vpt, kGenBlock, grid, 0, a.band_rows};
  }
  return e;
}

SlicedPlan choose_sliced(uint64_t streams, uint64_t rows, int device, bool may_split) {
  SlicedPlan p;
  const uint64_t tiles = (streams + kSlicedTile - 1) / kSlicedTile;
  // A partly filled last tile costs as much as a full one, and the other kernel
  // has smaller tiles: one tile at two thirds 118 / 109 us for 2^27 values and
  // 615 / 649 for 2^30, at 0.72 108 / 107 and 572 / 606, full 92 / 97 and 425 /
  // 551; two and three tiles the same within 4 %.
  if (streams * 3 < tiles * kSlicedTile * 2) return p;
  // Each tile pays for its states' way into bit planes and back, and small
  // launches need more blocks than there are tiles: us bit-sliced / best
  // checksum_kernel shape on GB300: 2^24 x 64 450 / 519, 2^22 x 64 144 / 147,
  // 2^20 x 128 88 / 96, 2^18 x 1024 130 / 166; below 2^27 values 2^18 x 256
  // 64 / 60, 65536 x 1024 65 / 60, 2^18 x 128 56 / 40.
  if (rows < 64 || streams * rows < (uint64_t(1) << 27)) return p;
  const uint64_t slots = static_cast<uint64_t>(device_sm_count(device)) *
                         static_cast<uint64_t>(occupancy(checksum_sliced_kernel_fn(), kSlicedBlock));
  const uint64_t waves = (tiles + slots - 1) / slots;
  const double whole = static_cast<double>(tiles) / static_cast<double>(waves * slots);  // share of the slots in use
  p.blocks = static_cast<uint32_t>(std::min(tiles, uint64_t(0x7fffffff)));
  if (!may_split || whole > 0.97) return p;
  // The fewest quanta per tile (each has its jump tables, one block's work) that
  // leave the longest run within 3 % of the mean; at least 16 rows each.
  double best = whole;
  for (uint64_t nq = 2; nq <= std::min<uint64_t>(rows / 16, kMaxBands); ++nq) {
    const uint64_t q = (rows + nq - 1) / nq;
    if ((rows + q - 1) / q != nq) continue;
    const uint64_t blocks = std::min(slots, tiles * nq);
    const uint64_t longest = (tiles * nq + blocks - 1) / blocks;
    const double use = static_cast<double>(tiles) * static_cast<double>(rows) /
                       (static_cast<double>(longest) * static_cast<double>(q) * static_cast<double>(slots));
    if (use <= best) continue;
    best = use;
    p.blocks = static_cast<uint32_t>(blocks);
    p.quantum_rows = q;
    if (use > 0.97) break;
  }
  return p;
}

cudaError_t launch_checksum_sliced(const RowsLaunch &a, const SlicedPlan &plan, uint64_t *row_xor, uint64_t *row_sum,
                                   cudaStream_t st, LaunchInfo *info) {
  if (!plan.blocks || (a.band_rows && !a.jump)) return cudaErrorInvalidValue;
  RowsLaunch args = a;
  unsigned long long *rx = reinterpret_cast<unsigned long long *>(row_xor);
  unsigned long long *rs = reinterpret_cast<unsigned long long *>(row_sum);
  void *params[] = {&args, &rx, &rs};
  cudaError_t e = cudaLaunchKernel(checksum_sliced_kernel_fn(), dim3(plan.blocks), dim3(kSlicedBlock), params, 0, st);
  if (e == cudaSuccess) {
    count_launch();
    *info = {RNG_KERNEL_SLICED, uint32_t(kSlicedTile / kSlicedBlock), kSlicedBlock, plan.blocks, 0, a.band_rows};
  }
  return e;
}

bool rows_vpt_supported(uint32_t vpt) { return rows_kernel_fn(vpt, 1, kStoreDefault, kGenBlock) != nullptr; }
bool rows_shape_supported(uint32_t vpt, uint32_t block) {
  return rows_kernel_fn(vpt ? vpt : 8, 1, kStoreStreaming, block ? block : kGenBlock) != nullptr;
}

bool batch_vpt_supported(uint32_t vpt) { return worklist_kernel_fn(vpt) != nullptr; }

int batch_blocks_per_sm(uint32_t vpt, uint32_t block) {
  const void *fn = worklist_kernel_fn(vpt);
  return fn ? occupancy(fn, block) : 0;
}

int batch_work_blocks_per_sm(uint32_t vpt, uint32_t bulk_nb) {
  if (bulk_nb) {
    const void *fn = batch_work_bulk_kernel_fn(vpt, bulk_nb);
    if (!fn) return 0;
    const size_t smem = rows_bulk_smem_bytes(vpt, bulk_nb);
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
      return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, static_cast<int>(kGenBlock), smem) != cudaSuccess || n < 1)
      n = 1;
    return n;
  }
  const void *fn = batch_work_kernel_fn(vpt);
  return fn ? occupancy(fn, kGenBlock) : 0;
}

cudaError_t launch_batch_work(const BatchWork *work, uint32_t n, uint32_t *counter, uint32_t vpt, uint32_t grid,
                              cudaStream_t st, uint32_t bulk_nb) {
  const void *fn = bulk_nb ? batch_work_bulk_kernel_fn(vpt, bulk_nb) : batch_work_kernel_fn(vpt);
  if (!fn) return cudaErrorInvalidValue;
  size_t smem = 0;
  if (bulk_nb) {
    smem = rows_bulk_smem_bytes(vpt, bulk_nb);
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  void *params[] = {&work, &n, &counter};
  cudaError_t e = cudaLaunchKernel(fn, dim3(grid), dim3(kGenBlock), params, smem, st);
  if (e == cudaSuccess) count_launch();
  return e;
}

cudaError_t launch_noalloc(const NoallocArgs &args, uint32_t tiles, cudaStream_t st) {
  void *params[] = {const_cast<NoallocArgs *>(&args)};
  const cudaError_t e = cudaLaunchKernel(noalloc_kernel_fn(), dim3(tiles), dim3(kGenBlock), params, 0, st);
  if (e == cudaSuccess) count_launch();
  return e;
}

cudaError_t launch_batch(const BatchInstance *inst, const BatchUnit *units, uint32_t n_units,
                         uint32_t *counter, uint32_t vpt, uint32_t block, uint32_t grid,
                         cudaStream_t st) {
  const void *fn = worklist_kernel_fn(vpt);
  if (!fn || block != kGenBlock) return cudaErrorInvalidValue;
  void *params[] = {&inst, &units, &n_units, &counter};
  cudaError_t e = cudaLaunchKernel(fn, dim3(grid), dim3(block), params, 0, st);
  if (e == cudaSuccess) count_launch();
  return e;
}

}  // namespace rngi
