// ck_launch.cuh -- host-side launch of the insert kernel, shared by the
// translation units that instantiate it (ck_insert_b1.cu, ck_insert_b4.cu,
// ck_insert_b8.cu: one bin size each, so they compile in parallel).
#pragma once
#include <cuda_runtime.h>

#include "ck.h"
#include "ck_kernels.cuh"
#include "ck_walk.cuh"
#include "ck_warp.cuh"

namespace ck {

// The host-side parameters of one insert launch (a table handle's fields).
struct InsertLaunch {
  const DevTable* dt;
  uint32_t block;
  int sm_count;
  bool overlap;          // the launch may start while its predecessor finishes (not upserts)
  uint64_t load_base;    // keys already in the table (the bins-viewed histogram's load)
  uint64_t max_threads;  // insertions in flight at most
};

using InsertFn = cudaError_t (*)(const InsertLaunch& l, const uint32_t* keys, const uint32_t* vals, uint64_t n,
                                 uint8_t* st, uint32_t* viewed, bool serial, uint32_t upsert, cudaStream_t s);

// The launch function for a policy, or nullptr (one definition per bin size).
InsertFn pick_insert_b1(uint32_t policy);
InsertFn pick_insert_b4(uint32_t policy, bool ghost);
InsertFn pick_insert_b8(uint32_t policy, bool ghost);
InsertFn pick_insert_warp_b4();  // BFS by a warp per search (CK_PARAM_SEARCH_WARP)
InsertFn pick_insert_warp_b8();

template <int B, int POL, bool GHOST>
cudaError_t launch_insert(const InsertLaunch& l, const uint32_t* keys, const uint32_t* vals, uint64_t n,
                          uint8_t* st, uint32_t* viewed, bool serial, uint32_t upsert, cudaStream_t s) {
  const DevTable& dt = *l.dt;
  const uint64_t load_base = l.load_base;
  if (serial) {
    k_insert<B, POL, GHOST, true><<<1, 1, 0, s>>>(dt, keys, vals, n, st, viewed, load_base, upsert);
    return cudaGetLastError();
  }
  const uint32_t block = l.block;
  // a step per lane (ck_walk.cuh), except upserts, which first look for the
  // key under claims
  const bool walk = !upsert;
  // An upsert's answer depends on the calls before it and the calls after it
  // on its own writes, so k_insert waits for its predecessor before it does
  // anything and lets nothing start beside it: only its launch overlaps (512
  // keys upserted, looked up and deleted: 25.2 us against 27.0 launched after it).
  const bool overlap = l.overlap && walk;
  const size_t shared = walk ? walk_shared<B, POL, GHOST>(block) : 0;
  if (shared) {  // on every launch: the attribute is the current device's
    const cudaError_t e = cudaFuncSetAttribute(k_insert_walk<B, POL, GHOST>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shared);
    if (e != cudaSuccess) return e;
  }
  // persistent launch: at most the blocks that fit on the GPU at once
  static int cached_block[2] = {0, 0}, cached_per_sm[2] = {0, 0};
  if (cached_block[walk] != (int)block) {
    int per_sm = 0;
    const cudaError_t e =
        walk ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_insert_walk<B, POL, GHOST>, block, shared)
             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_insert<B, POL, GHOST, false>, block, 0);
    if (e != cudaSuccess || per_sm < 1) per_sm = 1;
    cached_per_sm[walk] = per_sm;
    cached_block[walk] = (int)block;
  }
  uint64_t grid = (n + block - 1) / block;
  uint64_t resident = (uint64_t)cached_per_sm[walk] * l.sm_count;
  // A launch that may overlap the next leaves part of the GPU to it: its
  // blocks start while this launch's longest walks finish.  Walks keep 0.9 of
  // the resident blocks, rattle-kicking 0.8, measured when a warp still waited
  // for its longest walk (queue-kicking 10.18 ms against 10.45-10.50 with
  // every block, rattle-kicking 51.6 against 58.4); now the share hardly
  // shows (4- and 8-slot queue-kicking 6.41 / 0.84 ms against 6.39 / 0.87,
  // rattle-kicking 6.80 against 6.76).  Searches keep 0.7, which leaves L2 to
  // the table too: 2^22 x 4 to 0.95, sorted search 4.60 ms against 4.81 with
  // every block and 4.75 with 0.9, BFS 5.42 against 5.74 and 5.48, d = 4 sorted
  // search 6.32 against 6.56 and 6.47.  A limit the caller sets
  // (CK_PARAM_MAX_INFLIGHT) replaces this one.
  constexpr uint64_t tenths = (POL == P_QUEUE || POL == P_RANDOM) ? 9 : POL == P_RATTLE ? 8 : 7;
  if (overlap && l.max_threads == ~0ull) {
    const uint64_t most = resident * tenths / 10;
    resident = most > 0 ? most : 1;
  }
  if (grid > resident) grid = resident;
  uint64_t by_threads = l.max_threads / block;  // insertions in flight at once
  if (grid > by_threads) grid = by_threads > 0 ? by_threads : 1;
  if (dt.scratch) {
    uint64_t cap_blocks = (dt.n_searchers / SLAB) / ((block + SLAB - 1) / SLAB);
    if (grid > cap_blocks) grid = cap_blocks;
  }
  if (grid > 0x7FFFFFFFull) grid = 0x7FFFFFFFull;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = shared;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = l.overlap ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (walk) return cudaLaunchKernelEx(&cfg, k_insert_walk<B, POL, GHOST>, dt, keys, vals, n, st, viewed, load_base);
  return cudaLaunchKernelEx(&cfg, k_insert<B, POL, GHOST, false>, dt, keys, vals, n, st, viewed, load_base, upsert);
}

// The warp-search form of BFS (two-choice, no ghosts, concurrent only).
template <int B>
cudaError_t launch_insert_warp(const InsertLaunch& l, const uint32_t* keys, const uint32_t* vals, uint64_t n,
                               uint8_t* st, uint32_t* viewed, bool, uint32_t, cudaStream_t s) {
  const DevTable& dt = *l.dt;
  static int cached_per_sm = 0;
  if (cached_per_sm == 0) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_insert_warp<B>, WARP_BLOCK, 0) != cudaSuccess ||
        per_sm < 1)
      per_sm = 1;
    cached_per_sm = per_sm;
  }
  uint64_t grid = (n + WARP_BLOCK - 1) / WARP_BLOCK;
  const uint64_t resident = (uint64_t)cached_per_sm * l.sm_count;
  if (grid > resident) grid = resident;
  const uint64_t by_threads = l.max_threads / WARP_BLOCK;
  if (grid > by_threads) grid = by_threads > 0 ? by_threads : 1;
  const uint64_t cap_blocks = (dt.n_searchers / SLAB) / ((WARP_BLOCK + SLAB - 1) / SLAB);
  if (grid > cap_blocks) grid = cap_blocks;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(WARP_BLOCK);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = l.overlap ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_insert_warp<B>, dt, keys, vals, n, st, viewed, l.load_base);
}

// The two-choice policies for one bin size.
template <int B>
InsertFn pick_two_choice(uint32_t pol, bool ghost) {
  switch (pol) {
    case CK_RANDOM: return ghost ? launch_insert<B, P_RANDOM, true> : launch_insert<B, P_RANDOM, false>;
    case CK_BFS: return ghost ? launch_insert<B, P_BFS, true> : launch_insert<B, P_BFS, false>;
    case CK_SORTED: return ghost ? launch_insert<B, P_SORTED, true> : launch_insert<B, P_SORTED, false>;
    case CK_HYBRID: return ghost ? launch_insert<B, P_HYBRID, true> : launch_insert<B, P_HYBRID, false>;
    case CK_QUEUE: return ghost ? launch_insert<B, P_QUEUE, true> : launch_insert<B, P_QUEUE, false>;
    default: return nullptr;
  }
}

}  // namespace ck
