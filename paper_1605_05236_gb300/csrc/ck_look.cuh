// ck_look.cuh -- the first look at a batch's keys (two-choice tables without
// ghosts) and a block's counts, shared by the concurrent insert kernels.
//
// Most keys of a fill find a free slot in one of their bins.  A warp takes
// its keys 32 at a time, so that the loads of keys and the stores of statuses
// are coalesced, reads the slots of their bins -- no metadata word -- and
// places what it can by one compare-and-swap a key (place_direct).  The keys
// that found no room, or lost their slot to another thread, are kept by index
// in shared memory for the whole insertion, which a warp then enters with
// full lanes instead of the few of each 32 that need it.  Bound by the
// memory system: two random 128-byte lines a key (a random 32-byte miss
// moves its whole line) and the line written back.  Measured on one GB300,
// 2^20 keys a launch into an empty 2^24 x 4 table: 74 us against 90 with one
// key a thread through the whole insertion; two keys a lane in flight: 79.
#pragma once
#include "ck_search.cuh"

namespace ck {

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

// Randomised exponential backoff after a conflict: [w, 2w) ns with w =
// 64 << attempt, up to 32-64 us, so that long walks that keep meeting each
// other (small tables with most keys in flight) drift apart.  Measured on
// the 2^14 x 4 table with all 62,259 keys in flight at once (1.3 claim
// conflicts per key): capping w at 32 us rather than 1 ms fills it about 9%
// faster; the large fills do not change.
__device__ __forceinline__ uint32_t backoff_ns(uint32_t attempt, uint32_t key) {
  uint32_t w = 64u << (attempt < 9 ? attempt : 9);
  return w + (fmix32(key ^ attempt) & (w - 1));
}

__device__ __forceinline__ void backoff(uint32_t attempt, uint32_t key) { __nanosleep(backoff_ns(attempt, key)); }

// The bins-viewed histogram's bucket of a load of `at` keys.
__device__ __forceinline__ uint32_t load_bucket(uint64_t at, uint64_t total) {
  const uint64_t x = at * HIST_BUCKETS / total;
  return x < HIST_BUCKETS ? (uint32_t)x : HIST_BUCKETS - 1;
}

// What the insertions that ended in the lanes of `over` with st add up to (the
// whole warp calls; every lane gets the sums).
struct KeySums {
  uint32_t ok, failed, aborted, kicks, chain_max, viewed, viewed_all, aborts, reviews;
};
__device__ __forceinline__ KeySums sum_keys(bool over, const Ctx& c, int st, uint32_t aborts) {
  constexpr unsigned ALL = 0xFFFFFFFFu;
  KeySums s;
  const uint32_t k = over && st == ST_OK ? c.kicks : 0u;
  s.ok = __popc(__ballot_sync(ALL, over && st == ST_OK));
  s.failed = __popc(__ballot_sync(ALL, over && st == ST_FAILED));
  s.aborted = __popc(__ballot_sync(ALL, over)) - s.ok - s.failed;
  s.kicks = __reduce_add_sync(ALL, k);
  s.chain_max = __reduce_max_sync(ALL, k);
  s.viewed = __reduce_add_sync(ALL, over ? c.viewed - c.viewed0 : 0u);
  s.viewed_all = __reduce_add_sync(ALL, over ? c.viewed : 0u);
  s.aborts = __reduce_add_sync(ALL, over ? aborts : 0u);
  s.reviews = __reduce_add_sync(ALL, over ? c.reviews : 0u);
  return s;
}
// ... into a block's counters (shared memory) or a table's (global), by one
// lane
template <bool SHARED>
__device__ __forceinline__ void add_sums(unsigned long long* bc, const KeySums& s) {
  auto add = [&](int k, uint32_t x) {
    if (!x) return;
    if (SHARED) count_add(bc + k, x);
    else atomicAdd(bc + k, (unsigned long long)x);
  };
  add(C_INS_OK, s.ok);
  add(C_INS_FAILED, s.failed);
  add(C_INS_ABORTED, s.aborted);
  add(C_KICKS, s.kicks);
  if (s.chain_max) {
    if (SHARED) count_max(bc + C_CHAIN_MAX, s.chain_max);
    else atomicMax(bc + C_CHAIN_MAX, (unsigned long long)s.chain_max);
  }
  add(C_VIEWED, s.viewed);
  add(C_VIEWED_ALL, s.viewed_all);
  add(C_ABORTS, s.aborts);
  add(C_REVIEWS, s.reviews);
}

// A block's counts, in shared memory.
struct BlockTally {
  unsigned int views[HIST_BUCKETS], cnt[HIST_BUCKETS];  // bins viewed and keys, by load
  unsigned int chain[CHAIN_BUCKETS];
  unsigned long long bc[C_N];

  __device__ __forceinline__ void clear() {
    for (int i = threadIdx.x; i < HIST_BUCKETS; i += blockDim.x) views[i] = cnt[i] = 0;
    for (int i = threadIdx.x; i < CHAIN_BUCKETS; i += blockDim.x) chain[i] = 0;
    for (int i = threadIdx.x; i < C_N; i += blockDim.x) bc[i] = 0;
  }
  // a key's insertion ended with st, v bins viewed by its last attempt; what
  // every key adds to (insertions, bins viewed) the caller tallies
  __device__ __forceinline__ void key_done(const Ctx& c, int st, uint32_t aborts, uint32_t v, uint32_t bucket) {
    if (st == ST_OK) {
      if (c.kicks) {
        count_add(&bc[C_KICKS], c.kicks);
        count_max(&bc[C_CHAIN_MAX], c.kicks);
      }
      atomicAdd(&chain[chain_bucket(c.kicks)], 1u);
      if (c.ghosts_made) count_add(&bc[C_GHOSTS_MADE], c.ghosts_made);
      if (c.dup_evict) count_add(&bc[C_DUP_EVICT], c.dup_evict);
    } else {
      count_add(&bc[st == ST_FAILED ? C_INS_FAILED : C_INS_ABORTED], 1u);
    }
    if (aborts) count_add(&bc[C_ABORTS], aborts);
    if (c.reviews) count_add(&bc[C_REVIEWS], c.reviews);
    atomicAdd(&views[bucket], v);
    atomicAdd(&cnt[bucket], 1u);
  }
  // after a barrier, by the whole block: into the table's counters
  __device__ __forceinline__ void flush(const DevTable& t) {
    if (threadIdx.x == 0) {
      for (int k = 0; k < C_N; k++) {
        if (!bc[k]) continue;
        if (k == C_CHAIN_MAX) atomicMax(t.counters + k, bc[k]);
        else atomicAdd(t.counters + k, bc[k]);
      }
      // size and live ghosts follow from the counts above
      if (bc[C_INS_OK]) atomicAdd(t.counters + C_SIZE, bc[C_INS_OK]);
      long long dg = (long long)bc[C_GHOSTS_MADE] - (long long)bc[C_DUP_EVICT];
      if (dg) atomicAdd(t.counters + C_LIVE_GHOSTS, (unsigned long long)dg);
    }
    unsigned long long* hist = t.counters + C_N;
    for (int i = threadIdx.x; i < HIST_BUCKETS; i += blockDim.x) {
      if (cnt[i]) {
        atomicAdd(hist + i, (unsigned long long)views[i]);
        atomicAdd(hist + HIST_BUCKETS + i, (unsigned long long)cnt[i]);
      }
    }
    for (int i = threadIdx.x; i < CHAIN_BUCKETS; i += blockDim.x)
      if (chain[i]) atomicAdd(t.counters + CHAIN_HIST + i, (unsigned long long)chain[i]);
  }
};

// One lane's look at a key: placed (true) in a free slot it sees, or not;
// `views`: the bins viewed, `lost`: the slot was taken meanwhile (an attempt
// given up on a conflict).  Queue-kicking reads both bins and takes the less
// full one (b0 on ties); the other policies take b0's first free slot, else
// b1's, and fetch b1 only where b0 has none.  The searches count both bins as
// viewed either way, as their definition does.
template <int B, int POL>
__device__ __forceinline__ bool look_place(const DevTable& t, uint32_t key, uint32_t val, uint32_t& views,
                                           bool& lost) {
  uint32_t b0, b1;
  bins2(t, key, b0, b1);
  View<B> v;
  load_slots<B>(t, b0, v);
  uint32_t g0, g1 = 0;
  views = 2;
  lost = false;
  if (POL == P_QUEUE) {
    View<B> v1;
    load_slots<B>(t, b1, v1);
    g0 = empty_mask<B>(v);
    g1 = empty_mask<B>(v1);
    if (__popc(g0) >= __popc(g1)) g1 = 0;
    else g0 = 0;
  } else {
    g0 = empty_mask<B>(v);
    if (!g0) {
      load_slots<B>(t, b1, v);
      g1 = empty_mask<B>(v);
    } else if (POL == P_RANDOM) {
      views = 1;
    }
  }
  if (!(g0 | g1)) return false;
  const bool placed = cas_slot(t.slots + (uint64_t)(g0 ? b0 : b1) * B + lowest(g0 ? g0 : g1), EMPTY,
                               ((uint64_t)key << 32) | val);
  lost = !placed;
  return placed;
}

// A block's keys: the next index of its range, and per warp the keys looked
// at that found no room.
struct LookState {
  unsigned long long next;
  uint64_t left[8][64];
  uint32_t n_left[8];
  uint32_t bucket;       // the histogram bucket of the block's first keys ...
  uint64_t bucket_end;   // ... up to this index

  __device__ __forceinline__ void begin(const DevTable& t, uint64_t lo, uint64_t load_base) {
    if (threadIdx.x < 8) n_left[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
      next = lo;
      bucket = load_bucket(load_base + lo, t.total_slots);
      const uint64_t end = ((uint64_t)(bucket + 1) * t.total_slots + HIST_BUCKETS - 1) / HIST_BUCKETS;
      bucket_end = bucket == HIST_BUCKETS - 1 ? ~0ull : end - load_base;
    }
  }

  // One look at 32 new keys from `base` (those below hi), by a whole warp.
  template <int B, int POL>
  __device__ __forceinline__ uint32_t look(const DevTable& t, const uint32_t* __restrict__ keys,
                                           const uint32_t* __restrict__ vals, uint8_t* status, uint32_t* viewed_out,
                                           uint64_t base, uint64_t hi, uint64_t load_base, uint32_t nl,
                                           BlockTally& bt) {
    const uint64_t j = base + lane_id();
    const bool on = j < hi;
    const uint32_t key = on ? __ldcs(keys + j) : RESERVED_KEY;
    const uint32_t val = on ? __ldcs(vals + j) : 0u;
    uint32_t views = 0;
    bool lost = false;
    const bool placed = key != RESERVED_KEY && look_place<B, POL>(t, key, val, views, lost);
    const bool invalid = on && key == RESERVED_KEY;
    if (placed || invalid) {
      if (status) status[j] = (uint8_t)(invalid ? ST_INVALID : ST_OK);
      if (viewed_out) viewed_out[j] = invalid ? 0u : views;
    }
    const unsigned pm = __ballot_sync(0xFFFFFFFFu, placed), lm = __ballot_sync(0xFFFFFFFFu, lost);
    if (pm) {
      const uint32_t n = __popc(pm);
      const uint32_t sum = POL == P_RANDOM ? __reduce_add_sync(0xFFFFFFFFu, placed ? views : 0u) : 2 * n;
      const bool one = base + 32 <= bucket_end;  // the block's first bucket: one add for the warp
      if (lane_id() == 0) {
        count_add(&bt.bc[C_INS_OK], n);
        count_add(&bt.bc[C_VIEWED], sum);
        count_add(&bt.bc[C_VIEWED_ALL], sum);
        atomicAdd(&bt.chain[0], n);
        if (one) {
          atomicAdd(&bt.views[bucket], sum);
          atomicAdd(&bt.cnt[bucket], n);
        }
      }
      if (!one && placed) {
        const uint32_t b = load_bucket(load_base + j, t.total_slots);
        atomicAdd(&bt.views[b], views);
        atomicAdd(&bt.cnt[b], 1u);
      }
    }
    if (lm) {
      const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, lost ? views : 0u);
      if (lane_id() == 0) {
        count_add(&bt.bc[C_ABORTS], __popc(lm));
        count_add(&bt.bc[C_VIEWED_ALL], sum);
      }
    }
    const bool rest = on && !placed && !invalid;
    const unsigned rm = __ballot_sync(0xFFFFFFFFu, rest);
    if (rest) left[threadIdx.x >> 5][nl + __popc(rm & ((1u << lane_id()) - 1))] = j;
    return nl + __popc(rm);
  }

  // Keys for the lanes of `idle` (called by the whole warp): `got` is set to
  // the key's index, where one is left that needs the whole insertion.
  // False: the block's range is done, and so is the warp's list.
  template <int B, int POL>
  __device__ __forceinline__ bool take(const DevTable& t, const uint32_t* __restrict__ keys,
                                       const uint32_t* __restrict__ vals, uint8_t* status, uint32_t* viewed_out,
                                       uint64_t hi, uint64_t load_base, unsigned idle, BlockTally& bt,
                                       uint64_t& got) {
    const uint32_t wp = threadIdx.x >> 5, lane = lane_id(), want = __popc(idle);
    uint32_t nl = n_left[wp];
    bool more = true;
    while (nl < want) {
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(&next, 32ull);
      base = __shfl_sync(0xFFFFFFFFu, base, 0);
      if (base >= hi) {
        more = false;
        break;
      }
      nl = look<B, POL>(t, keys, vals, status, viewed_out, base, hi, load_base, nl, bt);
    }
    __syncwarp();
    const uint32_t give = nl < want ? nl : want, r = __popc(idle & ((1u << lane) - 1));
    if (((idle >> lane) & 1u) && r < give) got = left[wp][nl - give + r];
    __syncwarp();
    if (lane == 0) n_left[wp] = nl - give;
    __syncwarp();
    return more || nl > give;
  }
};

}  // namespace ck
