// ck_multi.cu -- the batched form: many independent two-choice cuckoo tables
// of uneven sizes filled in one persistent launch.
//
// Each table is a full table (slots, metadata, counters) of its own and is
// filled with the per-insertion code of the single-table path (the kick-out
// policies of Sec. 3-7 with claim flags and back-to-front chains, Sec. 8), so
// a key set gives the same key->value map per table either way.  What the
// batched form changes is scheduling.  The keys of all tables are cut into
// tiles, listed a group of tables that fits L2 at a time.  Walks
// (k_multi_walk: queue-kicking and random kicking): each warp takes pieces of
// 512 keys from the list, and its lanes walk in tables of their own, one launch
// for the 4-slot tables and one for the 8-slot ones.  With ghosts
// (k_multi_insert): each block takes a tile, and its threads the tile's keys.
// Small tables no longer leave the GPU idle and 4096 launches become one or
// two.  The reference path, ck_multi_insert_per_table, launches the
// single-table kernel once per table.
#include <cuda_runtime.h>

#include <cstring>
#include <new>
#include <vector>

#include "ck.h"
#include "ck_kernels.cuh"
#include "ck_walk.cuh"

using namespace ck;

// per-table path: the single-table launcher of ck_lib.cu
int ck_internal_launch_insert(const DevTable& dt, uint32_t block, int sm_count, const uint32_t* keys,
                              const uint32_t* vals, uint64_t n, uint8_t* status, cudaStream_t s,
                              uint64_t max_threads);

namespace {

constexpr size_t ALIGN = 256;
__host__ __device__ constexpr size_t align_up(size_t x) { return (x + ALIGN - 1) / ALIGN * ALIGN; }

struct Tile {
  uint32_t table;
  uint32_t pad;
  uint64_t lo, hi;  // key range in the shared key/value arrays
};

constexpr uint32_t MULTI_LONG_PLANS = 1024;
// Tables filled together.  Measured on 4096 tables (9.3 GB, 1.07e9 keys): 8
// and 16 MiB 90.0 ms, 32 MiB 90.4, 64 MiB 90.8, all tables at once 107.1.
constexpr size_t WINDOW_BYTES = 16u << 20;

}  // namespace

struct ck_multi {
  uint32_t n_tables;
  uint32_t policy;
  std::vector<ck_multi_desc> desc;
  std::vector<DevTable> host_tables;  // host copies of the device descriptors
  DevTable* d_tables;
  Tile* d_tiles;
  unsigned long long* d_tile_ctr;
  uint8_t* buf;
  size_t bytes;
  uint32_t n_tiles, n_tiles4;  // all, and those of 4-slot tables (first in the list)
  uint32_t tile;
  uint32_t block;
  uint32_t blocks_per_sm;  // 0: as many as fit
  uint32_t cap;
  int sm_count;
  cudaStream_t last;
  std::vector<size_t> table_off;  // byte offset of each table's slots
  size_t pool_off, busy_off, tables_off, tiles_off, ctr_off;
};

namespace {

struct MultiLayout {
  std::vector<size_t> off;  // per table: slots; meta and counters follow
  size_t tables, tiles, ctr, busy, pool, total;
  uint32_t n_tiles;
};

size_t table_bytes(const ck_multi_desc& d) {
  size_t b = align_up(d.bins * d.slots_per_bin * sizeof(uint64_t));
  b += align_up(d.bins * sizeof(uint32_t));
  b += align_up(COUNTER_WORDS * sizeof(uint64_t));
  return b;
}

uint32_t count_tiles(const ck_multi_desc* d, uint32_t n, uint32_t tile) {
  uint64_t t = 0;
  for (uint32_t i = 0; i < n; i++) t += (d[i].n_keys + tile - 1) / tile;
  return (uint32_t)t;
}

bool desc_ok(const ck_multi_desc* d, uint32_t n) {
  if (!d || n == 0) return false;
  for (uint32_t i = 0; i < n; i++) {
    if (d[i].bins < 2 || d[i].bins >= (1ull << 32)) return false;
    if (d[i].slots_per_bin != 4 && d[i].slots_per_bin != 8) return false;
  }
  return true;
}

// The tile list is sized for the smallest tile the autotuner may pick.
constexpr uint32_t MIN_TILE = 256;

MultiLayout multi_layout(const ck_multi_desc* d, uint32_t n) {
  MultiLayout L;
  size_t off = 0;
  L.off.resize(n);
  for (uint32_t i = 0; i < n; i++) {
    L.off[i] = off;
    off += table_bytes(d[i]);
  }
  L.tables = off;
  off = align_up(off + (size_t)n * sizeof(DevTable));
  L.n_tiles = count_tiles(d, n, MIN_TILE);
  L.tiles = off;
  off = align_up(off + (size_t)L.n_tiles * sizeof(Tile));
  L.ctr = off;
  off = align_up(off + (n + 1) * sizeof(unsigned long long));
  L.busy = off;
  off = align_up(off + MULTI_LONG_PLANS * sizeof(uint32_t));
  L.pool = off;
  off = align_up(off + (size_t)MULTI_LONG_PLANS * LONG_REGION);
  L.total = off;
  return L;
}

// Persistent batched insert (ghost policies): blocks pull tiles, threads pull
// keys.
template <int POL, bool GHOST>
__global__ void __launch_bounds__(256, 4) k_multi_insert(const DevTable* __restrict__ tables,
                                                      const Tile* __restrict__ tiles, uint32_t n_tiles,
                                                      unsigned long long* tile_ctr,
                                                      const uint32_t* __restrict__ keys,
                                                      const uint32_t* __restrict__ vals,
                                                      uint8_t* __restrict__ status) {
  __shared__ unsigned long long s_next, s_hi;
  __shared__ uint32_t s_tile, s_table;
  __shared__ unsigned long long bc[C_N];
  PlanStore<MAX_CHAIN> store;
  for (;;) {
    if (threadIdx.x == 0) {
      unsigned long long k = atomicAdd(tile_ctr, 1ull);
      s_tile = k < n_tiles ? (uint32_t)k : n_tiles;
      if (k < n_tiles) {
        Tile tl = tiles[k];
        s_table = tl.table;
        s_next = tl.lo;
        s_hi = tl.hi;
      }
    }
    for (int i = threadIdx.x; i < C_N; i += blockDim.x) bc[i] = 0;
    __syncthreads();
    if (s_tile >= n_tiles) break;
    const DevTable t = tables[s_table];
    const unsigned long long hi = s_hi;
    uint32_t ok = 0, failed = 0, aborted = 0, viewed = 0, viewed_all = 0, kicks = 0;  // per tile
    uint32_t aborts = 0, chain_max = 0, ghosts = 0, dupev = 0;
    for (;;) {
      const uint64_t i = take_index(&s_next);
      if (i >= hi) break;
      uint32_t key = keys[i];
      if (key == RESERVED_KEY) {
        if (status) status[i] = ST_INVALID;
        continue;
      }
      Ctx c;
      c.key = key;
      c.krec = ((uint64_t)key << 32) | vals[i];
      c.viewed = 0;
      c.reviews = 0;
      int st = t.B == 4 ? insert_one<4, POL, GHOST>(t, c, nullptr, aborts, store.e, MAX_CHAIN, true)
                        : insert_one<8, POL, GHOST>(t, c, nullptr, aborts, store.e, MAX_CHAIN, true);
      if (st == ST_OK) {
        ok++;
        kicks += c.kicks;
        chain_max = max(chain_max, c.kicks);
        ghosts += c.ghosts_made;
        dupev += c.dup_evict;
      } else if (st == ST_FAILED) {
        failed++;
      } else {
        aborted++;
      }
      viewed += c.viewed - c.viewed0;
      viewed_all += c.viewed;
      if (status) status[i] = (uint8_t)st;
    }
    if (ok) count_add(&bc[C_INS_OK], ok);
    if (failed) count_add(&bc[C_INS_FAILED], failed);
    if (aborted) count_add(&bc[C_INS_ABORTED], aborted);
    if (viewed) count_add(&bc[C_VIEWED], viewed);
    if (viewed_all) count_add(&bc[C_VIEWED_ALL], viewed_all);
    if (kicks) count_add(&bc[C_KICKS], kicks);
    if (aborts) count_add(&bc[C_ABORTS], aborts);
    if (ghosts) count_add(&bc[C_GHOSTS_MADE], ghosts);
    if (dupev) count_add(&bc[C_DUP_EVICT], dupev);
    if (chain_max) count_max(&bc[C_CHAIN_MAX], chain_max);
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 0; k < C_N; k++) {
        if (!bc[k]) continue;
        if (k == C_CHAIN_MAX) atomicMax(t.counters + k, bc[k]);
        else atomicAdd(t.counters + k, bc[k]);
      }
      if (bc[C_INS_OK]) atomicAdd(t.counters + C_SIZE, bc[C_INS_OK]);
      long long dg = (long long)bc[C_GHOSTS_MADE] - (long long)bc[C_DUP_EVICT];
      if (dg) atomicAdd(t.counters + C_LIVE_GHOSTS, (unsigned long long)dg);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------
// walks (tables without ghosts): lanes of a warp in tables of their own
// ------------------------------------------------------------------
// A warp takes pieces of SUB_TILE keys from the queue and gives its lanes the
// keys that found no room (ck_look.cuh); a lane goes on to the next piece's
// keys, in whichever table they are, when its walk ends, so no lane waits for
// a tile's longest walk and a piece can be small, which keeps the tables in
// work few enough for L2.  A warp keeps the counts of the tables it works on
// in shared memory and adds them to a table's counters when another takes
// the place.  4- and 8-slot tables have a launch each.
//
// Bound by latency (L2 round trips of looks and kicks), not by L2 or DRAM
// rates.  Measured, clear and fill of 4096 tables (9.3 GB, 1.07e9 keys) from a
// graph: 61 ms against 90 with a block a tile and an insertion a thread; 151
// with the counts added to the tables' counters per 32 keys (a few lines that
// every warp adds to); pieces of 256 / 512 / 1024 keys 72.7 / 64.8 / 61.1,
// with the queue asked a piece ahead 512 / 1024 / 2048: 61.2 / 62.2 / 70.7;
// 128 registers against 80: 60.9 against 62.2.
constexpr uint32_t SUB_TILE = 512;
// Tiles are listed in parts of at most LIST_TILE keys, the pieces of a part
// counted from its number in the queue: pieces past the end of a short part
// are taken and dropped.  4096 tables of 800 to 48,000 keys, tiles of 2^22 keys:
// 3.36 ms against 34.6 with a tile a part (8192 pieces for each table), 30.4
// with a block a tile; tiles of 4096: 3.25.
constexpr uint32_t LIST_TILE = 4096;
constexpr uint32_t NO_TABLE = 0xFFFFFFFFu;

struct PieceList {  // per warp, in shared memory
  uint64_t left[64];     // keys without room ...
  uint32_t left_t[64];   // ... and their tables
  uint64_t next, hi;     // the current piece's keys that were not looked at
  uint32_t table, n_left;
  uint32_t sums_of[4];   // counts of table sums_of[e] (e: its index mod 4)
  KeySums sums[4];
};

// Lane 0 of a warp: the counts in place e to their table's counters.
__device__ __forceinline__ void flush_sums(PieceList& pl, const DevTable* tables, uint32_t e) {
  if (pl.sums_of[e] == NO_TABLE) return;
  unsigned long long* ct = tables[pl.sums_of[e]].counters;
  add_sums<false>(ct, pl.sums[e]);
  if (pl.sums[e].ok) atomicAdd(ct + C_SIZE, (unsigned long long)pl.sums[e].ok);
}

// Lane 0 of a warp: the warp's counts of `table`.
__device__ __forceinline__ KeySums& sums_for(PieceList& pl, const DevTable* tables, uint32_t table) {
  const uint32_t e = table & 3u;
  if (pl.sums_of[e] != table) {
    flush_sums(pl, tables, e);
    pl.sums_of[e] = table;
    pl.sums[e] = KeySums{0, 0, 0, 0, 0, 0, 0, 0, 0};
  }
  return pl.sums[e];
}

template <int B, int POL>
struct TileKeys {
  DevTable t;  // the lane's table (the fields that differ, over the launch's common ones)
  const DevTable* tables;
  const Tile* tiles;
  uint64_t n_pieces;
  uint32_t per_tile;  // pieces a tile of the list
  unsigned long long* ctr;
  const uint32_t *keys, *vals;
  uint8_t* status;
  PieceList& pl;
  bool more;
  unsigned long long ahead;  // lane 0: the queue's next piece
  uint64_t i;
  uint32_t key, val, tab_of;  // the lane's key, its value and its table's index

  __device__ __forceinline__ const DevTable& table() const { return t; }

  static __device__ __forceinline__ void enter(DevTable& d, const DevTable& s) {
    d.slots = s.slots;
    d.meta = s.meta;
    d.n_bins = s.n_bins;
    d.bin_mask = s.bin_mask;
    d.bin_inv = s.bin_inv;
    if (POL == P_RANDOM) d.rng_seed = s.rng_seed;
  }

  // The warp's next piece; false: the queue is empty.  The queue's answer is
  // asked for a piece ahead, and the piece's keys and values are brought to
  // L2 (a line a lane).
  __device__ __forceinline__ bool next_piece() {
    for (;;) {
      const unsigned long long k = __shfl_sync(0xFFFFFFFFu, ahead, 0);
      if (k >= n_pieces) return false;
      if (lane_id() == 0) ahead = atomicAdd(ctr, 1ull);
      const Tile tl = tiles[k / per_tile];
      const uint64_t lo = tl.lo + (k % per_tile) * SUB_TILE, hi = min(tl.hi, lo + SUB_TILE);
      if (lo >= hi) continue;
      for (uint64_t j = lo + 32 * lane_id(); j < hi; j += 32 * 32) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(keys + j));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(vals + j));
      }
      if (lane_id() == 0) {
        pl.table = tl.table;
        pl.next = lo;
        pl.hi = hi;
      }
      __syncwarp();
      return true;
    }
  }

  __device__ __forceinline__ bool take(unsigned idle) {
    const uint32_t lane = lane_id(), want = __popc(idle);
    uint32_t nl = pl.n_left;
    while (nl < want) {
      if (pl.next >= pl.hi && !next_piece()) {
        more = false;
        break;
      }
      const uint64_t j = pl.next + lane;
      const uint32_t tab = pl.table;
      const bool on = j < pl.hi;
      const uint32_t k = on ? __ldcs(keys + j) : RESERVED_KEY, v = on ? __ldcs(vals + j) : 0u;
      DevTable d = t;
      enter(d, tables[tab]);
      uint32_t views = 0;
      bool lost = false;
      const bool placed = k != RESERVED_KEY && look_place<B, POL>(d, k, v, views, lost);
      const bool invalid = on && k == RESERVED_KEY;
      if ((placed || invalid) && status) status[j] = (uint8_t)(invalid ? ST_INVALID : ST_OK);
      const unsigned pm = __ballot_sync(0xFFFFFFFFu, placed), lm = __ballot_sync(0xFFFFFFFFu, lost);
      const uint32_t seen = __reduce_add_sync(0xFFFFFFFFu, placed ? views : 0u);
      const uint32_t wasted = lm ? __reduce_add_sync(0xFFFFFFFFu, lost ? views : 0u) : 0u;
      if (lane == 0) {
        KeySums& s = sums_for(pl, tables, tab);
        s.ok += __popc(pm);
        s.viewed += seen;
        s.viewed_all += seen + wasted;
        s.aborts += __popc(lm);
      }
      const bool rest = on && !placed && !invalid;
      const unsigned rm = __ballot_sync(0xFFFFFFFFu, rest);
      if (rest) {
        const uint32_t at = nl + __popc(rm & ((1u << lane) - 1));
        pl.left[at] = j;
        pl.left_t[at] = tab;
      }
      nl += __popc(rm);
      __syncwarp();
      if (lane == 0) pl.next += 32;
      __syncwarp();
    }
    const uint32_t give = nl < want ? nl : want, r = __popc(idle & ((1u << lane) - 1));
    const bool got = ((idle >> lane) & 1u) && r < give;
    if (got) {
      i = pl.left[nl - give + r];
      tab_of = pl.left_t[nl - give + r];
      enter(t, tables[tab_of]);
      key = __ldcs(keys + i);
      val = __ldcs(vals + i);
    }
    __syncwarp();
    if (lane == 0) pl.n_left = nl - give;
    __syncwarp();
    more = more || nl > give;
    return got;
  }

  __device__ __forceinline__ void done(bool over, const Ctx& c, int st, uint32_t aborts) {
    if (over && status) status[i] = (uint8_t)st;
    for (unsigned m = __ballot_sync(0xFFFFFFFFu, over); m;) {  // a table at a time
      const uint32_t tab = __shfl_sync(0xFFFFFFFFu, tab_of, __ffs(m) - 1);
      const bool in = over && tab_of == tab;
      const KeySums k = sum_keys(in, c, st, aborts);
      if (lane_id() == 0) {
        KeySums& s = sums_for(pl, tables, tab);
        s.ok += k.ok;
        s.failed += k.failed;
        s.aborted += k.aborted;
        s.kicks += k.kicks;
        s.chain_max = max(s.chain_max, k.chain_max);
        s.viewed += k.viewed;
        s.viewed_all += k.viewed_all;
        s.aborts += k.aborts;
        s.reviews += k.reviews;
      }
      m &= ~__ballot_sync(0xFFFFFFFFu, in);
    }
  }
};

template <int B, int POL>
__global__ void __launch_bounds__(256, 2) k_multi_walk(DevTable common, const DevTable* __restrict__ tables,
                                                       const Tile* __restrict__ tiles, uint64_t n_pieces,
                                                       uint32_t per_tile, unsigned long long* ctr,
                                                       const uint32_t* __restrict__ keys,
                                                       const uint32_t* __restrict__ vals,
                                                       uint8_t* __restrict__ status) {
  __shared__ PieceList pl[8];
  PieceList& mine = pl[threadIdx.x >> 5];
  if (lane_id() == 0) {
    mine.next = mine.hi = 0;
    mine.n_left = 0;
    for (int e = 0; e < 4; e++) mine.sums_of[e] = NO_TABLE;
  }
  __syncwarp();
  PlanStore<MAX_CHAIN> store;
  TileKeys<B, POL> src{common, tables, tiles, n_pieces, per_tile, ctr, keys, vals, status, mine, true, 0, 0,
                       0, 0, 0};
  if (lane_id() == 0) src.ahead = atomicAdd(ctr, 1ull);
  walk_keys<B, POL, false>(src, store.e);
  if (lane_id() == 0)
    for (uint32_t e = 0; e < 4; e++) flush_sums(mine, tables, e);
}

// Lookups across tables: key i belongs to table tab[i].
__global__ void __launch_bounds__(256) k_multi_lookup(const DevTable* __restrict__ tables,
                                                      const uint32_t* __restrict__ tab,
                                                      const uint32_t* __restrict__ keys, uint64_t n,
                                                      uint32_t* __restrict__ vals_out,
                                                      uint8_t* __restrict__ found_out) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const DevTable& t = tables[tab[i]];
    uint32_t key = keys[i];
    uint32_t val = 0;
    bool f = false;
    if (key != RESERVED_KEY) {
      uint32_t b0, b1;
      bins2(t, key, b0, b1);
      if (t.B == 4) {
        uint64_t s0[4], s1[4];
        load_bin_nc<4>(t, b0, s0);
        load_bin_nc<4>(t, b1, s1);
        f = match_bin<4>(s0, key, val);
        if (!f) f = match_bin<4>(s1, key, val);
      } else {
        uint64_t s0[8], s1[8];
        load_bin_nc<8>(t, b0, s0);
        load_bin_nc<8>(t, b1, s1);
        f = match_bin<8>(s0, key, val);
        if (!f) f = match_bin<8>(s1, key, val);
      }
    }
    if (vals_out) vals_out[i] = val;
    if (found_out) found_out[i] = (uint8_t)f;
  }
}

// The launches of one batched insertion, and the blocks of each that fit on
// an SM.  Ghost policies: one launch of k_multi_insert over all tiles; the
// others: k_multi_walk over the tiles of the 4-slot tables, then of the
// 8-slot ones.
template <class K>
int blocks_that_fit(K kernel, uint32_t block) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, 0) != cudaSuccess || per_sm < 1) return 1;
  return per_sm;
}

unsigned grid_of(const ck_multi* m, int fit, uint64_t most) {
  int per_sm = fit;
  if (m->blocks_per_sm && (int)m->blocks_per_sm < per_sm) per_sm = (int)m->blocks_per_sm;
  const uint64_t g = (uint64_t)per_sm * m->sm_count;
  return (unsigned)(g < most ? g : most > 0 ? most : 1);
}

template <int POL>
void launch_ghost(const ck_multi* m, const uint32_t* k, const uint32_t* v, uint8_t* st, cudaStream_t s) {
  const unsigned grid = grid_of(m, blocks_that_fit(k_multi_insert<POL, true>, m->block), m->n_tiles);
  k_multi_insert<POL, true><<<grid, m->block, 0, s>>>(m->d_tables, m->d_tiles, m->n_tiles, m->d_tile_ctr, k, v, st);
}

template <int B, int POL>
void launch_walk(const ck_multi* m, const uint32_t* k, const uint32_t* v, uint8_t* st, cudaStream_t s) {
  const uint32_t first = B == 4 ? 0 : m->n_tiles4, n = B == 4 ? m->n_tiles4 : m->n_tiles - m->n_tiles4;
  if (!n) return;
  const uint32_t per_tile = ((m->tile < LIST_TILE ? m->tile : LIST_TILE) + SUB_TILE - 1) / SUB_TILE;
  const uint64_t pieces = (uint64_t)n * per_tile;
  const uint32_t warps = m->block / 32;
  const unsigned grid = grid_of(m, blocks_that_fit(k_multi_walk<B, POL>, m->block), (pieces + warps - 1) / warps);
  k_multi_walk<B, POL><<<grid, m->block, 0, s>>>(m->host_tables[0], m->d_tables, m->d_tiles + first, pieces, per_tile,
                                                 m->d_tile_ctr + (B == 4 ? 0 : 1), k, v, st);
}

bool launch_multi(const ck_multi* m, const uint32_t* k, const uint32_t* v, uint8_t* st, cudaStream_t s) {
  const bool g = (m->policy & CK_GHOST) != 0;
  switch (m->policy & 0xFF) {
    case CK_RANDOM:
      if (g) return launch_ghost<P_RANDOM>(m, k, v, st, s), true;
      launch_walk<4, P_RANDOM>(m, k, v, st, s);
      launch_walk<8, P_RANDOM>(m, k, v, st, s);
      return true;
    case CK_QUEUE:
      if (g) return launch_ghost<P_QUEUE>(m, k, v, st, s), true;
      launch_walk<4, P_QUEUE>(m, k, v, st, s);
      launch_walk<8, P_QUEUE>(m, k, v, st, s);
      return true;
    default: return false;
  }
}

// Build the tile list for the current tile size and upload it: the tiles of
// the 4-slot tables, then those of the 8-slot ones.  The tables of a kind are
// taken in groups of about WINDOW_BYTES, in order, and the tiles of a
// group round-robin over its tables (tile r of each, then tile r + 1): the
// tables being filled stay in L2 from their first tile to their last, and
// each keeps only a part of its tiles in flight, so its load grows in order.
// For walks a tile is listed in parts of LIST_TILE keys.
void add_tiles(std::vector<Tile>& tiles, const ck_multi_desc* desc, uint32_t n_tables, uint32_t slots,
               uint32_t tile, uint32_t part) {
  std::vector<uint32_t> group;
  size_t bytes = 0;
  auto flush = [&]() {
    bool any = true;
    for (uint64_t r = 0; any; r++) {
      any = false;
      for (const uint32_t i : group) {
        const ck_multi_desc& d = desc[i];
        const uint64_t lo = r * tile;
        if (lo >= d.n_keys) continue;
        any = true;
        const uint64_t hi = lo + tile < d.n_keys ? lo + tile : d.n_keys;
        for (uint64_t a = lo; a < hi; a += part)
          tiles.push_back({i, 0, d.key_offset + a, d.key_offset + (a + part < hi ? a + part : hi)});
      }
    }
    group.clear();
    bytes = 0;
  };
  for (uint32_t i = 0; i < n_tables; i++) {
    if (desc[i].slots_per_bin != slots) continue;
    const size_t b = table_bytes(desc[i]);
    if (bytes + b > WINDOW_BYTES) flush();
    group.push_back(i);
    bytes += b;
  }
  flush();
}

int build_tiles(ck_multi* m, cudaStream_t s) {
  std::vector<Tile> tiles;
  tiles.reserve(count_tiles(m->desc.data(), m->n_tables, m->tile));
  const uint32_t part = (m->policy & CK_GHOST) ? m->tile : LIST_TILE;
  add_tiles(tiles, m->desc.data(), m->n_tables, 4, m->tile, part);
  m->n_tiles4 = (uint32_t)tiles.size();
  add_tiles(tiles, m->desc.data(), m->n_tables, 8, m->tile, part);
  m->n_tiles = (uint32_t)tiles.size();
  if (cudaMemcpyAsync(m->d_tiles, tiles.data(), tiles.size() * sizeof(Tile), cudaMemcpyHostToDevice, s) !=
      cudaSuccess)
    return CK_ECUDA;
  return cudaStreamSynchronize(s) == cudaSuccess ? CK_OK : CK_ECUDA;
}

// Empty every table and zero its counters, in one launch: block (i, y) takes
// every gridDim.y-th piece of table i.  A write pass over the tables (bound by
// DRAM).  Three memsets a table took 19 ms more on 4096 tables, replayed from
// a graph (126.2 ms for clear and fill against 107.1).
constexpr unsigned CLEAR_PARTS = 16;

__device__ __forceinline__ void fill16(void* p, uint64_t bytes, uint32_t v) {  // p and bytes: multiples of 16
  uint4* q = static_cast<uint4*>(p);
  const uint4 x = make_uint4(v, v, v, v);
  for (uint64_t i = (uint64_t)blockIdx.y * blockDim.x + threadIdx.x; i < bytes / 16; i += CLEAR_PARTS * blockDim.x) q[i] = x;
}

__global__ void __launch_bounds__(256) k_multi_clear(const DevTable* __restrict__ tables) {
  const DevTable& t = tables[blockIdx.x];
  // each part is followed by padding up to a multiple of 256 bytes
  fill16(t.slots, align_up(t.total_slots * sizeof(uint64_t)), 0xFFFFFFFFu);
  fill16(t.meta, align_up(t.n_bins * sizeof(uint32_t)), 0u);
  fill16(t.counters, align_up(COUNTER_WORDS * sizeof(uint64_t)), 0u);
}

int clear_tables(ck_multi* m, cudaStream_t s) {
  k_multi_clear<<<dim3(m->n_tables, CLEAR_PARTS), 256, 0, s>>>(m->d_tables);
  m->last = s;
  return cudaGetLastError() == cudaSuccess ? CK_OK : CK_ECUDA;
}

}  // namespace

extern "C" {

size_t ck_multi_required_bytes(const ck_multi_desc* h_desc, uint32_t n_tables) {
  if (!desc_ok(h_desc, n_tables)) return 0;
  return multi_layout(h_desc, n_tables).total;
}

int ck_multi_create_on(ck_multi** out, void* dev_buf, size_t bytes, const ck_multi_desc* h_desc, uint32_t n_tables,
                       uint32_t policy, uint64_t seed, void* stream) {
  if (!out) return CK_EINVAL;
  *out = nullptr;
  if (!desc_ok(h_desc, n_tables)) return CK_EINVAL;
  uint32_t pol = policy & 0xFF;
  if ((policy & ~0x1FFu) != 0 || (pol != CK_RANDOM && pol != CK_QUEUE)) return CK_ENOTSUP;
  if (!dev_buf || (reinterpret_cast<uintptr_t>(dev_buf) % ALIGN) != 0) return CK_EINVAL;
  MultiLayout L = multi_layout(h_desc, n_tables);
  if (bytes < L.total) return CK_ENOMEM;
  ck_multi* m = new (std::nothrow) ck_multi();
  if (!m) return CK_ENOMEM;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  m->n_tables = n_tables;
  m->policy = policy;
  m->desc.assign(h_desc, h_desc + n_tables);
  m->buf = static_cast<uint8_t*>(dev_buf);
  m->bytes = bytes;
  m->tile = 4096;
  m->block = 128;
  m->blocks_per_sm = 0;
  m->cap = 500;
  m->last = s;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    delete m;
    return CK_ECUDA;
  }
  m->d_tables = reinterpret_cast<DevTable*>(m->buf + L.tables);
  m->d_tiles = reinterpret_cast<Tile*>(m->buf + L.tiles);
  m->d_tile_ctr = reinterpret_cast<unsigned long long*>(m->buf + L.ctr);
  uint32_t* busy = reinterpret_cast<uint32_t*>(m->buf + L.busy);
  uint8_t* pool = m->buf + L.pool;
  m->host_tables.resize(n_tables);
  for (uint32_t i = 0; i < n_tables; i++) {
    const ck_multi_desc& d = h_desc[i];
    DevTable& t = m->host_tables[i];
    std::memset(&t, 0, sizeof(t));
    uint8_t* base = m->buf + L.off[i];
    size_t so = align_up(d.bins * d.slots_per_bin * sizeof(uint64_t));
    size_t mo = so + align_up(d.bins * sizeof(uint32_t));
    t.slots = reinterpret_cast<uint64_t*>(base);
    t.meta = reinterpret_cast<uint32_t*>(base + so);
    t.counters = reinterpret_cast<unsigned long long*>(base + mo);
    t.scratch = nullptr;
    t.long_scratch = pool;
    t.long_busy = busy;
    t.slab_busy = nullptr;
    t.n_bins = d.bins;
    t.total_slots = d.bins * d.slots_per_bin;
    t.rng_seed = seed + i;
    t.bin_mask = (d.bins & (d.bins - 1)) == 0 ? (uint32_t)(d.bins - 1) : 0u;
    t.bin_inv = inverse_of(d.bins);
    t.B = d.slots_per_bin;
    t.d = 2;
    t.policy = pol;
    t.ghost = (policy & CK_GHOST) ? 1 : 0;
    t.cap = m->cap;
    t.max_retries = 1024;
    t.ordered_writes = 0;
    t.spawn_k = 1;
    t.n_searchers = 0;
    t.n_long = MULTI_LONG_PLANS;
    t.hash_family = 0;
    t.seeds[0] = 0x9E3779B9u;
    t.seeds[1] = 0x85EBCA6Bu;
    t.seeds[2] = 0xC2B2AE35u;
    t.seeds[3] = 0x27D4EB2Fu;
  }
  int rc = CK_OK;
  if (cudaMemcpyAsync(m->d_tables, m->host_tables.data(), n_tables * sizeof(DevTable), cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaMemsetAsync(busy, 0, MULTI_LONG_PLANS * sizeof(uint32_t), s) != cudaSuccess)
    rc = CK_ECUDA;
  if (rc == CK_OK) rc = clear_tables(m, s);
  if (rc == CK_OK) rc = build_tiles(m, s);
  if (rc != CK_OK) {
    delete m;
    return rc;
  }
  *out = m;
  return CK_OK;
}

int ck_multi_set_param(ck_multi* m, int key, int64_t value) {
  if (!m) return CK_EINVAL;
  switch (key) {
    case CK_MULTI_TILE:
      if (value < MIN_TILE || value > (1 << 22)) return CK_EINVAL;
      m->tile = (uint32_t)value;
      return build_tiles(m, m->last);
    case CK_MULTI_BLOCK:
      if (value != 64 && value != 128 && value != 256) return CK_EINVAL;
      m->block = (uint32_t)value;
      return CK_OK;
    case CK_MULTI_BLOCKS_PER_SM:
      if (value < 0 || value > 32) return CK_EINVAL;
      m->blocks_per_sm = (uint32_t)value;
      return CK_OK;
    case CK_MULTI_CHAIN_CAP: {
      if (value < 1 || value > LONG_CHAIN - 8) return CK_EINVAL;
      m->cap = (uint32_t)value;
      for (auto& t : m->host_tables) t.cap = m->cap;
      if (cudaMemcpyAsync(m->d_tables, m->host_tables.data(), m->n_tables * sizeof(DevTable), cudaMemcpyHostToDevice,
                          m->last) != cudaSuccess)
        return CK_ECUDA;
      return CK_OK;
    }
    default:
      return CK_EINVAL;
  }
}

int ck_multi_insert(ck_multi* m, const uint32_t* d_keys, const uint32_t* d_vals, uint8_t* d_status, void* stream) {
  if (!m || !d_keys || !d_vals) return CK_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(m->d_tile_ctr, 0, 2 * sizeof(unsigned long long), s) != cudaSuccess) return CK_ECUDA;
  if (!launch_multi(m, d_keys, d_vals, d_status, s)) return CK_ENOTSUP;
  m->last = s;
  return cudaGetLastError() == cudaSuccess ? CK_OK : CK_ECUDA;
}

int ck_multi_insert_per_table(ck_multi* m, const uint32_t* d_keys, const uint32_t* d_vals, uint8_t* d_status,
                              void* stream) {
  if (!m || !d_keys || !d_vals) return CK_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  for (uint32_t i = 0; i < m->n_tables; i++) {
    const ck_multi_desc& d = m->desc[i];
    if (!d.n_keys) continue;
    // in flight at once: at most 1/16 of the table's slots (one block at
    // least), the operating range of the claim protocol (Sec. 8 runs a few
    // threads on a large table); launches of different tables overlap
    uint64_t max_threads = d.bins * d.slots_per_bin / 16;
    if (max_threads < m->block) max_threads = m->block;
    int rc = ck_internal_launch_insert(m->host_tables[i], m->block, m->sm_count, d_keys + d.key_offset,
                                       d_vals + d.key_offset, d.n_keys, d_status ? d_status + d.key_offset : nullptr,
                                       s, max_threads);
    if (rc != CK_OK) return rc;
  }
  m->last = s;
  return CK_OK;
}

int ck_multi_lookup(ck_multi* m, const uint32_t* d_table, const uint32_t* d_keys, uint64_t n, uint32_t* d_vals_out,
                    uint8_t* d_found, void* stream) {
  if (!m) return CK_EINVAL;
  if (n == 0) return CK_OK;
  if (!d_table || !d_keys) return CK_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  uint64_t g = (n + 255) / 256;
  if (g > 0x7FFFFFFFull) g = 0x7FFFFFFFull;
  k_multi_lookup<<<(unsigned)g, 256, 0, s>>>(m->d_tables, d_table, d_keys, n, d_vals_out, d_found);
  m->last = s;
  return cudaGetLastError() == cudaSuccess ? CK_OK : CK_ECUDA;
}

int ck_multi_table_stats(ck_multi* m, uint32_t table, ck_stats_t* out) {
  if (!m || !out || table >= m->n_tables) return CK_EINVAL;
  unsigned long long c[C_N];
  if (cudaStreamSynchronize(m->last) != cudaSuccess) return CK_ECUDA;
  if (cudaMemcpy(c, m->host_tables[table].counters, sizeof(c), cudaMemcpyDeviceToHost) != cudaSuccess) return CK_ECUDA;
  std::memset(out, 0, sizeof(*out));
  out->inserts_ok = c[C_INS_OK];
  out->inserts_failed = c[C_INS_FAILED];
  out->inserts_aborted = c[C_INS_ABORTED];
  out->bins_viewed = c[C_VIEWED];
  out->kicks = c[C_KICKS];
  out->chain_max = c[C_CHAIN_MAX];
  out->aborts = c[C_ABORTS];
  out->ghost_pairs_made = c[C_GHOSTS_MADE];
  out->dup_evictions = c[C_DUP_EVICT];
  out->size = c[C_SIZE];
  out->live_ghosts = c[C_LIVE_GHOSTS];
  out->conflict_views = c[C_REVIEWS];
  out->bins_viewed_all = c[C_VIEWED_ALL];
  out->total_slots = m->host_tables[table].total_slots;
  out->load = out->total_slots ? (double)out->size / (double)out->total_slots : 0.0;
  uint64_t ins = out->inserts_ok + out->inserts_failed + out->inserts_aborted;
  out->bins_viewed_per_insert = ins ? (double)out->bins_viewed / (double)ins : 0.0;
  out->aborts_per_insert = ins ? (double)out->aborts / (double)ins : 0.0;
  return CK_OK;
}

int ck_multi_stats(ck_multi* m, ck_stats_t* out) {
  if (!m || !out) return CK_EINVAL;
  ck_stats_t sum;
  std::memset(&sum, 0, sizeof(sum));
  uint64_t chain_max = 0;
  for (uint32_t i = 0; i < m->n_tables; i++) {
    ck_stats_t s;
    int rc = ck_multi_table_stats(m, i, &s);
    if (rc != CK_OK) return rc;
    sum.inserts_ok += s.inserts_ok;
    sum.inserts_failed += s.inserts_failed;
    sum.inserts_aborted += s.inserts_aborted;
    sum.bins_viewed += s.bins_viewed;
    sum.kicks += s.kicks;
    sum.aborts += s.aborts;
    sum.ghost_pairs_made += s.ghost_pairs_made;
    sum.dup_evictions += s.dup_evictions;
    sum.size += s.size;
    sum.live_ghosts += s.live_ghosts;
    sum.conflict_views += s.conflict_views;
    sum.bins_viewed_all += s.bins_viewed_all;
    sum.total_slots += s.total_slots;
    if (s.chain_max > chain_max) chain_max = s.chain_max;
  }
  sum.chain_max = chain_max;
  sum.load = sum.total_slots ? (double)sum.size / (double)sum.total_slots : 0.0;
  uint64_t ins = sum.inserts_ok + sum.inserts_failed + sum.inserts_aborted;
  sum.bins_viewed_per_insert = ins ? (double)sum.bins_viewed / (double)ins : 0.0;
  sum.aborts_per_insert = ins ? (double)sum.aborts / (double)ins : 0.0;
  *out = sum;
  return CK_OK;
}

int ck_multi_export(ck_multi* m, uint32_t table, uint64_t* h_slots, uint32_t* h_meta) {
  if (!m || table >= m->n_tables) return CK_EINVAL;
  if (cudaStreamSynchronize(m->last) != cudaSuccess) return CK_ECUDA;
  const DevTable& t = m->host_tables[table];
  if (h_slots && cudaMemcpy(h_slots, t.slots, t.total_slots * sizeof(uint64_t), cudaMemcpyDeviceToHost) != cudaSuccess)
    return CK_ECUDA;
  if (h_meta && copy_meta_out(t, h_meta) != cudaSuccess) return CK_ECUDA;
  return CK_OK;
}

int ck_multi_clear(ck_multi* m, void* stream) {
  if (!m) return CK_EINVAL;
  return clear_tables(m, reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"

// A captured fill of a batched form: the graph and its executable.
struct ck_graph {
  cudaGraph_t graph;
  cudaGraphExec_t exec;
  ck_multi* m;
};

extern "C" {

int ck_multi_capture(ck_multi* m, const uint32_t* d_keys, const uint32_t* d_vals, uint8_t* d_status,
                     uint32_t flags, void* stream, ck_graph** out) {
  if (!out) return CK_EINVAL;
  *out = nullptr;
  if (!m || !d_keys || !d_vals) return CK_EINVAL;
  if (flags & ~(uint32_t)(CK_MULTI_CAPTURE_CLEAR | CK_MULTI_CAPTURE_PER_TABLE)) return CK_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  bool own = false;
  if (!s) {  // the legacy default stream cannot be captured: use a stream of our own
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return CK_ECUDA;
    own = true;
  }
  const cudaStream_t last = m->last;
  int rc = CK_OK;
  if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) rc = CK_ECUDA;
  if (rc == CK_OK) {
    if (flags & CK_MULTI_CAPTURE_CLEAR) rc = clear_tables(m, s);
    if (rc == CK_OK)
      rc = (flags & CK_MULTI_CAPTURE_PER_TABLE) ? ck_multi_insert_per_table(m, d_keys, d_vals, d_status, s)
                                                : ck_multi_insert(m, d_keys, d_vals, d_status, s);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(s, &g);  // always ends the capture, even after an error
    if (rc == CK_OK && (e != cudaSuccess || !g)) rc = CK_ECUDA;
    ck_graph* h = nullptr;
    if (rc == CK_OK) {
      h = new (std::nothrow) ck_graph();
      if (!h) rc = CK_ENOMEM;
    }
    if (rc == CK_OK && cudaGraphInstantiate(&h->exec, g, 0) != cudaSuccess) rc = CK_ECUDA;
    if (rc == CK_OK) {
      h->graph = g;
      h->m = m;
      *out = h;
    } else {
      if (g) cudaGraphDestroy(g);
      delete h;
      cudaGetLastError();
    }
  }
  m->last = last;  // nothing ran yet: the handle's readers keep waiting where they did
  if (own) cudaStreamDestroy(s);
  return rc;
}

int ck_graph_launch(ck_graph* g, void* stream) {
  if (!g) return CK_EINVAL;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaGraphLaunch(g->exec, s) != cudaSuccess) return CK_ECUDA;
  g->m->last = s;
  return CK_OK;
}

void ck_graph_destroy(ck_graph* g) {
  if (!g) return;
  cudaGraphExecDestroy(g->exec);
  cudaGraphDestroy(g->graph);
  delete g;
}

void ck_multi_destroy(ck_multi* m) {
  if (!m) return;
  if (m->last) cudaStreamSynchronize(m->last);
  delete m;
}

}  // extern "C"
