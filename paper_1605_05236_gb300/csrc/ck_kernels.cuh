// ck_kernels.cuh -- the bulk kernels of the GB300 cuckoo table: insert
// (every policy), lookup and delete (Kuszmaul, arXiv:1605.05236, Sec. 1,
// Sec. 3-8), plus their per-batch counters.
#pragma once
#include "ck_look.cuh"

namespace ck {

template <int B, int POL, bool GHOST>
__device__ __forceinline__ int attempt_insert(const DevTable& t, Ctx& c, uint8_t* region) {
  if constexpr (B == 1) {
    if constexpr (POL == P_RATTLE) return insert_rattle(t, c);
    else if constexpr (POL == P_RANDOM) return insert_random_dary(t, c);
    else return insert_search_dary<POL>(t, c, region);
  } else if constexpr (POL == P_QUEUE) {
    return insert_queue<B, GHOST>(t, c);
  } else if constexpr (POL == P_BFS || POL == P_SORTED || POL == P_HYBRID) {
    return insert_search<B, POL, GHOST>(t, c, region);
  } else {
    return insert_random2<B, GHOST>(t, c);
  }
}

// One insertion with bounded retries after claim conflicts.  A chain that
// outgrows the local plan continues in a scratch plan.  retry_failed: in
// concurrent mode an attempt that ran out is made again (six times, 32 while
// it meets other insertions' claims): its path depended on their timing.
template <int B, int POL, bool GHOST>
__device__ __forceinline__ int insert_one(const DevTable& t, Ctx& c, uint8_t* region, uint32_t& aborts,
                                          uint64_t* local_e, int local_cap, bool retry_failed = false) {
  c.long_id = -1;
  c.big_id = -1;
  int st;
  uint32_t fails = 0;
  for (uint32_t attempt = 0;;) {
    c.attempt = attempt;
    c.kicks = 0;
    c.draws = 0;
    c.viewed0 = c.viewed;
    c.ghosts_made = 0;
    c.dup_evict = 0;
    c.foreign = 0;
    c.capped = 0;
    if (c.long_id < 0) {
      c.pe = local_e;
      c.pcap = local_cap;
    }
    c.pn = 0;
    st = attempt_insert<B, POL, GHOST>(t, c, region);
    bool undone = false;
    if (st == ST_OK) {
      if (commit<B>(t, c)) break;
      st = ST_CONFLICT;  // a slot no longer held what the plan expected: its writes were undone
      undone = true;
    }
    release_all(t, c, undone);
    if (st == ST_LONG) {  // a search path longer than the local plan
      if (c.long_id >= 0 || !grow_plan(t, c)) { st = c.long_id >= 0 ? ST_FAILED : ST_ABORTED; break; }
      continue;
    }
    // a walk or search that ran out is retried at most six times, or 32
    // times while it meets other insertions' claims on the way (they
    // finish meanwhile); then the key is FAILED
    const bool ran_out = st == ST_FAILED || (st == ST_CONFLICT && c.capped);
    if (ran_out) {
      if (!retry_failed || ++fails > (st == ST_FAILED ? 6u : 32u)) {
        st = ST_FAILED;
        break;
      }
      // a search out of budget tries again in a larger space (search_space)
      if (region && c.big_id < 0 && (POL == P_BFS || POL == P_SORTED || POL == P_HYBRID))
        c.big_id = take_big_space(t, c.key);
    } else {
      aborts++;
    }
    if (++attempt >= t.max_retries) { st = ST_ABORTED; break; }
    // a failed attempt waits longer before its retry: the walks and claims
    // of the insertions around it, which made it fail, finish meanwhile
    backoff(ran_out ? 6 + 2 * fails : attempt, c.key);
  }
  if (c.long_id >= 0) release_long(t, c.long_id);
  if (c.big_id >= 0) release_long(t, c.big_id);
  return st;
}

// ------------------------------------------------------------------
// deletes (Sec. 1): every copy goes, each under its claim flag (Sec. 8)
// ------------------------------------------------------------------
// The copies of a key that a delete or an overwrite holds claimed.
template <int B>
struct Copies {
  static constexpr int D = B == 1 ? 4 : 2;  // bins of a key at most
  uint32_t b[4];      // its bins
  uint32_t seen[D];   // their metadata words as read
  uint32_t slots[D];  // the copies: slots of each bin
  uint64_t rec;       // the record in them (every copy holds the same)
};

// The metadata words of a key's bins, all read before any of the bins'
// slots: a record that moves between the key's bins moves under its source's
// claim, whose release changes that bin's word, but the free slot it moves to
// need not be claimed (ck_walk.cuh), so both words have to be from before.
__device__ __forceinline__ void read_words(const DevTable& t, const uint32_t* b, uint32_t nb, uint32_t* seen) {
  for (uint32_t j = 0; j < nb; j++) seen[j] = ld_relaxed(t.meta + b[j]);
  fence_acquire();
}

// Drop the claims on the copies; `bump`: with a version bump.
template <int B>
__device__ __forceinline__ void drop_copies(const DevTable& t, const Copies<B>& k, bool bump) {
#pragma unroll
  for (int j = 0; j < Copies<B>::D; j++)
    if (k.slots[j]) red_relaxed(t.meta + k.b[j], (bump ? VER_ONE : 0u) - k.slots[j]);
}

// Find the key and claim the slots holding it.  1: claimed; 0: absent, which
// is reported only when the bins were seen unclaimed and unchanged across the
// read (unchanged_since); 2: a writer is in the way (nothing claimed).
template <int B>
__device__ __forceinline__ int claim_copies(const DevTable& t, uint32_t key, Copies<B>& k) {
  constexpr uint32_t CLAIM_BITS = (1u << B) - 1;
  constexpr int D = Copies<B>::D;
  const uint32_t nb = B == 1 ? t.d : 2u;
#pragma unroll
  for (int j = 0; j < D; j++) k.slots[j] = 0;
  read_words(t, k.b, nb, k.seen);
  bool conflict = false, any = false;
#pragma unroll
  for (int j = 0; j < D; j++) {
    if (j >= (int)nb || conflict) continue;
    View<B> v;
    load_slots<B>(t, k.b[j], v);
    uint32_t add = 0;
#pragma unroll
    for (int s = 0; s < B; s++) add |= (v.s[s] != EMPTY && key_of(v.s[s]) == key ? 1u : 0u) << s;
    if (!add) continue;
    const uint64_t r = slot_of<B>(v, lowest(add));
    conflict = (add & k.seen[j]) != 0 ||           // a writer holds it
               (any && r != k.rec) ||              // copies that differ: a writer is active
               !cas_acquire(t.meta + k.b[j], k.seen[j], k.seen[j] + add);
    if (conflict) continue;
    any = true;
    k.rec = r;
    k.slots[j] = add;
  }
  if (!conflict && any) return 1;
  if (!conflict && unchanged_since(t.meta, k.b, k.seen, nb, CLAIM_BITS)) return 0;
  drop_copies<B>(t, k, false);
  return 2;
}

// Replace the record in every claimed copy by `to`, each by a 64-bit
// compare-and-swap from the record seen when the copies were viewed: a
// claim validates a view through the metadata word only, and that word can
// come back to an earlier value.  If a copy no longer holds the record, the
// copies already replaced get it back, the claims are dropped and the call
// returns false.
template <int B>
__device__ __forceinline__ bool swap_copies(const DevTable& t, const Copies<B>& k, uint64_t to) {
  constexpr int D = Copies<B>::D;
  uint32_t done[D];
  bool ok = true;
#pragma unroll
  for (int j = 0; j < D; j++) {
    done[j] = 0;
    for (uint32_t m = k.slots[j]; m && ok; m &= m - 1) {
      ok = cas_slot(t.slots + (uint64_t)k.b[j] * B + lowest(m), k.rec, to);
      if (ok) done[j] |= m & (0u - m);
    }
  }
  if (ok) return true;
#pragma unroll
  for (int j = 0; j < D; j++)
    for (uint32_t m = done[j]; m; m &= m - 1) st_slot(t.slots + (uint64_t)k.b[j] * B + lowest(m), k.rec);
  fence_release();
  drop_copies<B>(t, k, true);
  return false;
}

// One delete: every copy claimed, cleared, released (a ghost pair has two).  A
// delete running beside insertions on another stream never misses a key that
// is being moved (claim_copies).  Slots claimed by a writer are waited out
// with backoff, at most DELETE_ATTEMPTS times (status 2).
//
// Bound by random accesses, of which a key found in its first or second bin
// needs six: two words, two bins, the claim and the slot's write (the
// release hits the line of the claim).  The copies are held as slot masks:
// kept as a list in local memory, 2^22 deletes in 2^24 x 4 at 0.95 and their
// insertion took 0.88 ms, against 0.79.
constexpr int DELETE_ATTEMPTS = 1024;

__device__ __forceinline__ void wait_for_writer(uint32_t attempt, uint32_t key) {
  const uint32_t w = 128u << (attempt < 13 ? attempt : 13);
  __nanosleep(w + (fmix32(key ^ attempt) & (w - 1)));
}

template <int B>
__device__ __forceinline__ int delete_one(const DevTable& t, uint32_t key, uint32_t& ghost_removed) {
  Copies<B> k;
  bins_of(t, key, k.b);
  for (int attempt = 0; attempt < DELETE_ATTEMPTS; attempt++) {
    const int r = claim_copies<B>(t, key, k);
    if (r == 0) return 0;
    if (r == 2 || !swap_copies<B>(t, k, EMPTY)) {
      wait_for_writer(attempt, key);
      continue;
    }
    fence_release();
    int dup_copies = 0;
#pragma unroll
    for (int j = 0; j < Copies<B>::D; j++) {
      const uint32_t m = k.slots[j];
      if (!m) continue;
      uint32_t delta = VER_ONE - m;
      if (B == 1) {
        delta -= rattle_of(k.seen[j]) << RATTLE_SHIFT;  // the bin forgets r(x)
      } else {
        const uint32_t dup = m & (k.seen[j] >> DUP_SHIFT);
        delta -= dup << DUP_SHIFT;                       // duplicate marks go too
        dup_copies += __popc(dup);
        if (t.policy == P_QUEUE) delta += HIT_ONE * __popc(m);  // fewer slots, the same hits
      }
      red_relaxed(t.meta + k.b[j], delta);
    }
    ghost_removed += dup_copies >= 2 ? 1 : 0;
    return 1;
  }
  return 2;
}

// Overwrite the value of a present key (CK_INS_UPSERT): claim every slot
// holding it (both copies of a ghost pair), store the new record, release
// with a version bump; the duplicate marks stay.  Returns 1 if updated, 0 if
// the key is absent (a miss proven as delete_one proves it), 2 if claimed
// slots were not released within DELETE_ATTEMPTS tries.
template <int B>
__device__ __forceinline__ int update_one(const DevTable& t, uint32_t key, uint64_t rec) {
  Copies<B> k;
  bins_of(t, key, k.b);
  for (int attempt = 0; attempt < DELETE_ATTEMPTS; attempt++) {
    const int r = claim_copies<B>(t, key, k);
    if (r == 0) return 0;
    if (r == 2 || !swap_copies<B>(t, k, rec)) {
      wait_for_writer(attempt, key);
      continue;
    }
    fence_release();
    drop_copies<B>(t, k, true);
    return 1;
  }
  return 2;
}

// Insert kernel, one insertion a thread from view to commit.  Serial mode
// (SERIAL, one thread): keys in batch order, one insertion in flight, a
// scratch-backed plan; this replays the paper's serial algorithms exactly.
// Concurrent mode runs upserts (the other concurrent insertions go a step per
// lane, ck_walk.cuh): each block takes a contiguous range of the batch and its
// threads pull keys from it, plans in local memory.
//
// Neither mode overlaps the launches around it (those of k_insert_walk do): an
// upsert must find the keys of the calls before it, what follows must find
// the upsert's, and a serial replay has one insertion in flight.  So there is
// no launch_dependents here, and the first thing done is the wait for the
// launch before.
// `load_base` is the number of keys the table held before this batch (for the
// histogram).
// Registers: at most 64 (4 blocks of 256 or 8 of 128 threads per SM) for
// most policies, 80 for 4-slot queue-kicking (3 blocks of 256).  Measured on
// one GB300, fill of 2^24 x 4 to 0.95: queue-kicking 10.36-10.52 ms at 80
// registers (no spills) vs 10.56-10.74 at 64 (92 bytes spilled); random
// kicking 25.1 ms at 80 vs 24.0-24.4 at 64: the kernel is bound by random
// accesses in flight, and only the queue kernel's spills cost more than the
// warps a larger register file takes away.
template <int B, int POL>
constexpr int insert_blocks_per_sm() { return (B == 4 && POL == P_QUEUE) ? 3 : 4; }

template <int B, int POL, bool GHOST, bool SERIAL>
__global__ void __launch_bounds__(256, insert_blocks_per_sm<B, POL>()) k_insert(DevTable t, const uint32_t* __restrict__ keys,
                                                const uint32_t* __restrict__ vals, uint64_t n,
                                                uint8_t* __restrict__ status,
                                                uint32_t* __restrict__ viewed_out, uint64_t load_base,
                                                uint32_t upsert) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ BlockTally bt;
  __shared__ unsigned long long s_next;  // next key of this block's range
  __shared__ int s_slab[SLABS_PER_BLOCK], s_long;
  bt.clear();
  // each block owns a contiguous range of the batch; its threads pull keys
  // from it one at a time, so a thread held up by a long chain does not
  // hold up the others
  const uint64_t per = (n + gridDim.x - 1) / gridDim.x;
  const uint64_t lo = min(n, (uint64_t)blockIdx.x * per), hi = min(n, lo + per);
  if (threadIdx.x == 0) {
    s_next = lo;
    const int need = (int)((blockDim.x + SLAB - 1) / SLAB);
    if (!t.scratch || !acquire_slabs(t, s_slab, need)) s_slab[0] = -1;
    s_long = SERIAL ? acquire_long(t, 0) : -1;
  }
  __syncthreads();

  PlanStore<SERIAL ? 1 : MAX_CHAIN> store;
  uint64_t* local_e = store.e;
  int local_cap = SERIAL ? 1 : MAX_CHAIN;
  bool usable = true;
  if (SERIAL) {
    if (s_long >= 0) {
      local_e = reinterpret_cast<uint64_t*>(t.long_scratch + (uint64_t)s_long * LONG_REGION);
      local_cap = LONG_CHAIN;
    } else {
      usable = false;
    }
  }
  uint8_t* region = slab_region(t, s_slab);
  if (t.scratch && !region) usable = false;

  // per-thread tallies of the counts every key adds to (32-bit: a thread
  // handles far fewer than 2^32 keys or bin views in one launch), flushed
  // into the block's 64-bit counters at the end; the rarer counts go to the
  // block's counters as they happen, which keeps them out of registers for
  // the whole loop
  uint32_t ok = 0, viewed = 0, viewed_all = 0;
  // Is key i to be inserted?  (If not, it was overwritten or refused.)
  auto inserts = [&](uint64_t i, Ctx& c) {
    c.key = keys[i];
    int r = 0;
    if (c.key != RESERVED_KEY) {
      c.krec = ((uint64_t)c.key << 32) | vals[i];
      // a present key is overwritten in place, not inserted again
      if (!upsert || (r = update_one<B>(t, c.key, c.krec)) == 0) return true;
      count_add(&bt.bc[r == 1 ? C_UPDATES : C_INS_ABORTED], 1u);
    }
    if (status) status[i] = (uint8_t)(r == 0 ? ST_INVALID : r == 1 ? ST_UPDATED : ST_ABORTED);
    if (viewed_out) viewed_out[i] = 0;
    return false;
  };
  // Each thread takes its indices for itself: one add a warp (by
  // __activemask) held threads up for one another, 5.7 ms against 3.6
  // (queue-kicking, 2^22 x 4 from 0.80 to 0.93, half the upserts present).
  // Searches in d-ary tables look on until each thread of a warp has an
  // insertion to do (sorted search, d = 4, 2^23 bins from 0.75 to 0.90: 7.1 ms
  // against 7.9); two-choice tables are 2-5% slower that way.
  constexpr bool LOOK_ON = B == 1 && POL != P_RANDOM && POL != P_RATTLE;
  for (;;) {
    Ctx c;
    uint64_t i;
    if constexpr (LOOK_ON) {
      while ((i = atomicAdd(&s_next, 1ull)) < hi)
        if (inserts(i, c)) break;
      if (i >= hi) break;
    } else {
      i = atomicAdd(&s_next, 1ull);
      if (i >= hi) break;
      if (!inserts(i, c)) continue;
    }
    c.viewed = c.viewed0 = 0;
    c.reviews = 0;
    uint32_t aborts = 0;
    // concurrent mode retries a failed attempt: other insertions moved records
    // meanwhile, so the next walk or search differs; the serial replay never
    // retries
    int st = usable ? insert_one<B, POL, GHOST>(t, c, region, aborts, local_e, local_cap, !SERIAL)
                    : (int)ST_ABORTED;
    // bins viewed by the attempt that was applied (or failed), and by all
    // attempts including those abandoned after claim conflicts
    uint32_t v_final = c.viewed - c.viewed0;
    viewed += v_final;
    viewed_all += c.viewed;
    if (status) status[i] = (uint8_t)st;
    if (viewed_out) viewed_out[i] = v_final;
    ok += st == ST_OK;
    bt.key_done(c, st, aborts, v_final, load_bucket(load_base + i, t.total_slots));
  }
  if constexpr (SERIAL) {
    count_add(&bt.bc[C_INS_OK], ok);
    count_add(&bt.bc[C_VIEWED], viewed);
    count_add(&bt.bc[C_VIEWED_ALL], viewed_all);
  } else {
    count_add_warp(&bt.bc[C_INS_OK], ok);
    count_add_warp(&bt.bc[C_VIEWED], viewed);
    count_add_warp(&bt.bc[C_VIEWED_ALL], viewed_all);
  }
  __syncthreads();
  bt.flush(t);
  if (threadIdx.x == 0) {
    release_slabs(t, s_slab);
    if (s_long >= 0) release_long(t, s_long);
  }
}

// ------------------------------------------------------------------
// lookups (Sec. 1: a present key sits in one of its d bins)
// ------------------------------------------------------------------

// Read-only 32-byte sector load through the non-coherent path: lookups run
// with no writer in flight on the table.
__device__ __forceinline__ void ld_bin4_nc(const uint64_t* p, uint64_t* s) {
  asm volatile("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];"
               : "=l"(s[0]), "=l"(s[1]), "=l"(s[2]), "=l"(s[3]) : "l"(p));
}

__device__ __forceinline__ uint64_t ld_slot_nc(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.global.nc.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}

template <int B>
__device__ __forceinline__ bool match_bin(const uint64_t* s, uint32_t key, uint32_t& val) {
  bool f = false;
#pragma unroll
  for (int q = 0; q < B; q++) {
    if (!f && key_of(s[q]) == key) { f = true; val = (uint32_t)s[q]; }
  }
  return f;
}

template <int B>
__device__ __forceinline__ void load_bin_nc(const DevTable& t, uint32_t bin, uint64_t* s) {
  const uint64_t* p = t.slots + (uint64_t)bin * B;
#pragma unroll
  for (int q = 0; q < B; q += 4) ld_bin4_nc(p + q, s + q);
}

// What a lookup launch adds to the table's counters.
__device__ __forceinline__ void count_lookups(const DevTable& t, uint32_t hits, uint32_t cnt) {
  __shared__ unsigned long long sh[2];
  if (threadIdx.x < 2) sh[threadIdx.x] = 0;
  __syncthreads();
  count_add_warp(&sh[0], hits);
  count_add_warp(&sh[1], cnt);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (sh[0]) atomicAdd(t.counters + C_LOOKUP_HITS, sh[0]);
    if (sh[1]) atomicAdd(t.counters + C_LOOKUPS, sh[1]);
  }
}

// Two-choice lookup: the first bin, and the second for keys not found there.
// Bound by random DRAM lines (a random miss moves a 128-byte line whatever
// part of it is read): 2^26 lookups, half of them hits, in a 2^24 x 4 table
// at 0.95 take 2.03 ms, 1.75 lines a lookup at 58 G lines/s of the 61 the
// gather probe reaches.
//
// 8-slot bins are read by pairs of lanes, half a bin each, one key of the
// pair after the other: the two 32-byte halves then travel as one access.
// Read by two instructions of one lane they cost two, though the line is the
// same.  20,000,003 lookups, 0 / 50 / 90% hits, 2^23 x 8 at 0.97 (512 MiB): 718
// / 614 / 532 us against 1142 / 942 / 793; 5,000,011 x 8 (320 MB): 625 / 538 /
// 477 against 790 / 654 / 559; 2^17 x 8 (8 MiB, in L2): 246 / 246 / 229 against
// 383 / 362 / 324; 2^16 lookups: the same.  Both keys of the pair in flight
// together take 40-48 registers instead of 32 and are slower (566 and 621 for
// 538).
template <int B>
__global__ void __launch_bounds__(256) k_lookup2(DevTable t, const uint32_t* __restrict__ keys, uint64_t n,
                                                 uint32_t* __restrict__ vals_out,
                                                 uint8_t* __restrict__ found_out) {
  uint32_t hits = 0, cnt = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t n32 = (n + 31) & ~31ull;  // whole warps: pairs of lanes work together
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n32; i += stride) {
    const uint32_t key = i < n ? __ldcs(keys + i) : RESERVED_KEY;
    uint32_t val = 0;
    bool f = false;
    uint32_t b0 = 0, b1 = 0;
    if (key != RESERVED_KEY) bins2(t, key, b0, b1);
    if constexpr (B == 8) {
      constexpr unsigned ALL = 0xFFFFFFFFu;
      const uint32_t half = threadIdx.x & 1u, even = threadIdx.x & 30u;
#pragma unroll
      for (uint32_t u = 0; u < 2; u++) {  // the even lane's key, then the odd lane's
        const uint32_t k = __shfl_sync(ALL, key, even + u);
        const bool on = k != RESERVED_KEY;
        uint32_t bin = __shfl_sync(ALL, b0, even + u), v = 0;
        uint64_t s[4];
        if (on) ld_bin4_nc(t.slots + (uint64_t)bin * 8 + half * 4, s);
        bool h = on && match_bin<4>(s, k, v);
        const bool other = __shfl_xor_sync(ALL, h, 1);
        bin = __shfl_sync(ALL, b1, even + u);
        if (on && !h && !other) {
          ld_bin4_nc(t.slots + (uint64_t)bin * 8 + half * 4, s);
          h = match_bin<4>(s, k, v);
        }
        const bool ph = __shfl_xor_sync(ALL, h, 1);
        const uint32_t pv = __shfl_xor_sync(ALL, v, 1);
        if (half == u) {  // stored twice: the lower half's copy, for either lane
          f = h || ph;
          val = h && (half == 0 || !ph) ? v : ph ? pv : 0u;
        }
      }
    } else if (key != RESERVED_KEY) {
      uint64_t s[B];
      load_bin_nc<B>(t, b0, s);
      f = match_bin<B>(s, key, val);
      if (!f) {
        load_bin_nc<B>(t, b1, s);
        f = match_bin<B>(s, key, val);
      }
    }
    if (i < n) {
      hits += f;
      cnt++;
      if (vals_out) __stcs(vals_out + i, val);
      if (found_out) __stcs(found_out + i, (uint8_t)f);
    }
  }
  count_lookups(t, hits, cnt);
}

// d-ary lookup: a bin is read only for keys not found in the ones before,
// which saves a DRAM line (a present key is in its second or third bin on
// average); with this many keys in flight the round trips do not show.  2^26
// bins, d = 4, 0.90 full, 2^24 lookups, 50 / 90% hits: 927 / 761 us against
// 1134 with all d bins fetched at once; 2^20 lookups 75 / 65 against 87; 2^16
// and fewer the same.
static __global__ void __launch_bounds__(256) k_lookup_dary(DevTable t, const uint32_t* __restrict__ keys, uint64_t n,
                                                     uint32_t* __restrict__ vals_out,
                                                     uint8_t* __restrict__ found_out) {
  uint32_t hits = 0, cnt = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    uint32_t key = __ldcs(keys + i);
    uint32_t val = 0;
    bool f = false;
    if (key != RESERVED_KEY) {
      uint32_t b[4];
      bins_of(t, key, b);
#pragma unroll
      for (int j = 0; j < 4; j++) {
        if (f || j >= (int)t.d) continue;
        const uint64_t r = ld_slot_nc(t.slots + b[j]);
        if (key_of(r) == key) { f = true; val = (uint32_t)r; }
      }
    }
    hits += f;
    cnt++;
    if (vals_out) __stcs(vals_out + i, val);
    if (found_out) __stcs(found_out + i, (uint8_t)f);
  }
  count_lookups(t, hits, cnt);
}

// The hit field of n bins' metadata words, for an export (sign 1: the bin's
// occupied slots added, which makes it queue-kicking's hit counter) and back
// (sign -1).  B is 4 or 8; in and out may be the same words.
static __global__ void __launch_bounds__(256) k_convert_hits(const uint64_t* slots, const uint32_t* in, uint32_t* out,
                                                             uint64_t n, uint32_t B, int sign) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b < n; b += stride) {
    uint32_t occupied = 0;
    for (uint32_t s = 0; s < B; s++) occupied += slots[b * B + s] != EMPTY;
    const uint32_t m = in[b];
    const uint32_t h = ((m >> HIT_SHIFT) + (uint32_t)sign * occupied) & 255u;
    out[b] = (m & ~(255u << HIT_SHIFT)) | (h << HIT_SHIFT);
  }
}

inline cudaError_t convert_hits(const DevTable& t, uint64_t first, uint64_t n, uint32_t* out, int sign) {
  const unsigned grid = (unsigned)(n < 256 * 4096 ? (n + 255) / 256 : 4096);
  k_convert_hits<<<grid, 256>>>(t.slots + first * t.B, t.meta + first, out, n, t.B, sign);
  return cudaGetLastError();
}

// Metadata words to host memory in the exported form (hit counters of
// queue-kicking tables), converted a part at a time in a buffer of its own:
// an export reads the table and writes nothing of it, so exports may run
// beside each other and beside lookups.  On the legacy default stream.
inline cudaError_t copy_meta_out(const DevTable& t, uint32_t* h_meta) {
  if (t.policy != P_QUEUE || t.B == 1)
    return cudaMemcpy(h_meta, t.meta, t.n_bins * sizeof(uint32_t), cudaMemcpyDeviceToHost);
  uint64_t part = t.n_bins < (1u << 22) ? t.n_bins : 1u << 22;  // 16 MiB at most, less where memory is short
  uint32_t* buf = nullptr;
  cudaError_t e;
  while ((e = cudaMalloc(&buf, part * sizeof(uint32_t))) == cudaErrorMemoryAllocation && part > 4096) {
    cudaGetLastError();
    part /= 2;
  }
  if (e != cudaSuccess) return e;
  for (uint64_t b = 0; b < t.n_bins && e == cudaSuccess; b += part) {
    const uint64_t n = t.n_bins - b < part ? t.n_bins - b : part;
    e = convert_hits(t, b, n, buf, 1);
    if (e == cudaSuccess) e = cudaMemcpy(h_meta + b, buf, n * sizeof(uint32_t), cudaMemcpyDeviceToHost);
  }
  cudaFree(buf);
  return e;
}

// Words as exported, back into the device's form (the slots are in place).
inline cudaError_t convert_meta_in(const DevTable& t) {
  if (t.policy != P_QUEUE || t.B == 1) return cudaSuccess;
  const cudaError_t e = convert_hits(t, 0, t.n_bins, t.meta, -1);
  return e == cudaSuccess ? cudaStreamSynchronize(nullptr) : e;  // callers may go on on another stream
}

template <int B>
__global__ void __launch_bounds__(256) k_delete(DevTable t, const uint32_t* __restrict__ keys, uint64_t n,
                                                uint8_t* __restrict__ found_out) {
  __shared__ unsigned long long bc[4];
  if (threadIdx.x < 4) bc[threadIdx.x] = 0;
  __syncthreads();
  uint32_t hits = 0, aborts = 0, ghosts = 0, cnt = 0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    uint32_t key = keys[i];
    int r = key == RESERVED_KEY ? 0 : delete_one<B>(t, key, ghosts);
    hits += r == 1;
    aborts += r == 2;
    cnt++;
    if (found_out) found_out[i] = (uint8_t)r;
  }
  count_add_warp(&bc[0], hits);
  count_add_warp(&bc[1], aborts);
  count_add_warp(&bc[2], ghosts);
  count_add_warp(&bc[3], cnt);
  __syncthreads();
  if (threadIdx.x == 0) {
    if (bc[0]) {
      atomicAdd(t.counters + C_DELETE_HITS, bc[0]);
      atomicAdd(t.counters + C_SIZE, 0ull - bc[0]);
    }
    if (bc[1]) atomicAdd(t.counters + C_DELETE_ABORTS, bc[1]);
    if (bc[2]) atomicAdd(t.counters + C_LIVE_GHOSTS, 0ull - bc[2]);
    if (bc[3]) atomicAdd(t.counters + C_DELETES, bc[3]);
  }
}

}  // namespace ck
