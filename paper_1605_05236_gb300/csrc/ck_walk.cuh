// ck_walk.cuh -- concurrent insertion by kick-out walks (queue-kicking and
// random kicking, two-choice tables without ghosts; Kuszmaul,
// arXiv:1605.05236, Sec. 1, Sec. 6, Sec. 8) with every lane of a warp at its
// own point of its own walk.
//
// What bounds the insertions of a nearly full table is chains of dependent
// round trips, and walks are uneven: near load 0.95 a key kicks five records
// on average and the longest of 32 keys about forty, so a warp that waits
// for its longest walk before it takes new keys keeps a fifth of its lanes
// busy.  Here a walk is a state (Walk) that advances one kick a step; a lane
// whose walk ends applies it and takes the next key while the others go on.
// The parts that end and begin walks cost several round trips and all lanes
// pass through them, so they run when most lanes wait for them (WAITERS), not
// for each.  Fill of 2^24 x 4 to 0.95 in 2^20-key batches: 6.33 ms against
// 9.27 with one insertion a lane from view to commit (k_insert) and 8.34 with
// the first look alone; its last launch (load 0.94) 0.88 ms against 1.45.
//
// The claims, the re-validation of moves and the order of writes are
// ck_insert.cuh's, with one difference: the free slot a chain ends in is not
// claimed.  Nothing moves out of it, so no reader's proof of a miss and no
// other plan rests on its claim, and the write that takes it is a
// compare-and-swap from empty anyway; the claim and its release were two
// more atomics on a metadata line the chain otherwise only reads.  The
// compare-and-swap is the chain's first write, made once the last claimed
// slot was read again and found as planned; if it fails, the walk views the
// bin again with nothing written.
#pragma once
#include "ck_look.cuh"

namespace ck {

constexpr int WALK = -1;  // the walk goes on
static_assert(WALK == SEARCHING && WALK == KICKING, "every unfinished insertion says so alike");

template <bool C, class X, class Y>
struct Choose { using type = X; };
template <class X, class Y>
struct Choose<false, X, Y> { using type = Y; };

template <int POL>
constexpr bool is_search_policy = POL == P_BFS || POL == P_SORTED || POL == P_HYBRID;

// A walk at a bin it has viewed, with the record c.held in hand.
template <int B>
struct Walk {
  uint32_t x;            // the bin
  int s;                 // random kicking: the slot to kick (-1: not drawn yet)
  uint32_t tries;        // views of x beyond the first
  View<B> v;             // x as viewed
  const uint64_t* pend;  // the slot claimed by the last kick, not read again yet (reread), or null
};

// The two bins of a new key: placed if there is room (ST_OK), else the walk's
// first bin is chosen.
template <int B, int POL>
__device__ __forceinline__ int walk_begin(const DevTable& t, Ctx& c, Walk<B>& w) {
  constexpr uint32_t FULL = (1u << B) - 1;
  c.held = c.krec;
  w.pend = nullptr;
  w.tries = 0;
  w.s = -1;
  if constexpr (POL == P_RATTLE) {
    w.s = 0;
    return WALK;
  }
  uint32_t b0, b1;
  bins2(t, c.key, b0, b1);
  View<B> v0, v1;
  load_view2_fast<B>(t, b0, b1, v0, v1);
  const uint32_t g0 = empty_mask<B>(v0), g1 = empty_mask<B>(v1);
  c.viewed += (POL == P_RANDOM && g0) ? 1 : 2;
  if (g0 | g1) {
    const bool first = POL == P_QUEUE ? __popc(g0) >= __popc(g1) : g0 != 0;
    return place_direct<B>(t, c, first ? b0 : b1, lowest(first ? g0 : g1)) ? (int)ST_OK : (int)ST_CONFLICT;
  }
  bool first;
  if (POL == P_QUEUE) {
    first = hit_of_full<B>(v0.m) <= hit_of_full<B>(v1.m);
  } else {  // first victim: uniform over the usable slots of b0 then b1
    const uint32_t e0 = FULL & ~claimed_mask<B>(v0), e1 = FULL & ~claimed_mask<B>(v1);
    const uint32_t n0 = __popc(e0), ne = n0 + __popc(e1);
    if (ne == 0) return ST_CONFLICT;
    const uint32_t idx = below(draw(t, c.key, c.draws++, c.attempt), ne);
    first = idx < n0;
    w.s = first ? nth_bit(e0, idx) : nth_bit(e1, idx - n0);
  }
  w.x = first ? b0 : b1;
  w.v.m = first ? v0.m : v1.m;
#pragma unroll
  for (int q = 0; q < B; q++) w.v.s[q] = first ? v0.s[q] : v1.s[q];
  return WALK;
}

// A step of rattle-kicking (insert_rattle, ck_insert.cuh, which the serial
// replay runs): one try, the record in hand at its bin h_{r mod d}, where
// w.s is r and c.draws counts the tries.  The bin's view and the re-read of
// the slot the kick before claimed go out together.
__device__ __forceinline__ int rattle_step(const DevTable& t, Ctx& c, Walk<1>& w) {
  if (c.draws == t.cap) return out_of_cap(c);
  c.draws++;
  if (int r = plan_room(t, c)) return r;
  uint32_t vb[4];
  bins_of(t, key_of(c.held), vb);
  const uint32_t j = (uint32_t)w.s % t.d;
  const uint32_t x = j == 0 ? vb[0] : j == 1 ? vb[1] : j == 2 ? vb[2] : vb[3];
  const uint32_t rc = w.s < 255 ? w.s + 1 : 255;
  w.s = (int)rc;
  const uint64_t chk = w.pend ? ld_slot(w.pend) : c.held;
  View<1> v;
  load_view_fast<1>(t, x, v);
  if (chk != c.held) return ST_CONFLICT;
  w.pend = nullptr;
  for (int k = 0;; k++) {
    if (claimed_mask<1>(v)) {
      // this chain's own bin: skipped, not viewed; another insertion's:
      // viewed and ignored (Sec. 8)
      if (k || !plan_has_bin(c, x)) {
        if (!k) c.viewed++;
        c.foreign = 1;
      }
      return WALK;
    }
    if (!k) c.viewed++;
    const uint32_t ry = rattle_of(v.m);
    if (v.s[0] == EMPTY) {
      if (claim(t, c, x, v.m, 0, K_MOVE, false, c.held, ry, rc)) return ST_OK;
    } else {
      if (t.tie_resident ? rc <= ry : rc < ry) return WALK;  // the resident stays
      if (claim(t, c, x, v.m, 0, K_MOVE, false, c.held, ry, rc)) {
        c.kicks++;
        c.held = v.s[0];
        w.s = (int)ry;
        w.pend = t.slots + x;
        return WALK;
      }
    }
    if (k == 3) return ST_CONFLICT;
    load_view_fast<1>(t, x, v);
    c.viewed++;
    c.reviews++;
  }
}

// One step at w.x: the free slot that ends the chain (ST_OK, and it is
// written), or one kick -- the claim of the victim, the view of the bin it
// moves to and the re-read of the slot the kick before claimed, in one round
// trip -- or another view of the bin after a lost race (WALK).
template <int B, int POL>
__device__ __forceinline__ int walk_step(const DevTable& t, Ctx& c, Walk<B>& w) {
  if constexpr (POL == P_RATTLE) return rattle_step(t, c, w);
  constexpr uint32_t FULL = (1u << B) - 1;
  const uint64_t chk = w.pend ? ld_slot(w.pend) : c.held;
  const uint32_t fm = empty_mask<B>(w.v);
  bool again = true;
  if (fm) {
    if (chk != c.held) return ST_CONFLICT;
    w.pend = nullptr;  // read again and as planned
    uint64_t* p = t.slots + (uint64_t)w.x * B + lowest(fm);
    if (cas_slot(p, EMPTY, c.held)) return ST_OK;
  } else {
    const uint32_t claimed = claimed_mask<B>(w.v);
    int s = w.s, jprev = -1;
    bool rev = false;
    if (POL == P_QUEUE) {
      // the record at slot h mod B, skipping slots another insertion holds;
      // a slot this chain already wrote is taken again, with the record the
      // chain put there
      const uint32_t own = claimed ? own_slots(c, w.x) : 0u;
      const uint32_t foreign = claimed & ~own;
      if (foreign) c.foreign = 1;
      s = first_from<B>(FULL & ~foreign, hit_of_full<B>(w.v.m) % B);
      if (s < 0) return dead_end(c);
      if (c.kicks == t.cap) return out_of_cap(c);
      rev = (own >> s) & 1u;
      if (rev) jprev = last_entry_for(c, w.x, (uint32_t)s);
    } else {
      if (c.kicks == t.cap) return ST_FAILED;
      if (s < 0) {  // uniform over the slots no chain holds
        const uint32_t e = FULL & ~claimed;
        if (!e) return claims_all_ours<B>(c, w.x, claimed) ? (int)ST_FAILED : (int)ST_CONFLICT;
        s = nth_bit(e, below(draw(t, c.key, c.draws++, c.attempt), __popc(e)));
        w.s = s;
      } else if ((claimed >> s) & 1u) {  // taken while the claim was tried
        return ST_CONFLICT;
      }
    }
    if (int r0 = plan_room(t, c)) return r0;
    const uint64_t victim = rev ? content_at(c, jprev) : slot_of<B>(w.v, s);
    const uint32_t xn = other_bin2(t, victim, w.x);
    View<B> vn;
    load_view_fast<B>(t, xn, vn);
    // (an entry of this kernel's plans holds the record its slot receives)
    if (rev ? claim_again(t, c, w.x, w.v.m, s, jprev, c.held)
            : claim(t, c, w.x, w.v.m, s, K_MOVE, POL == P_QUEUE, c.held)) {
      if (chk != c.held) return ST_CONFLICT;
      c.kicks++;
      // a slot the chain holds already carries the plan's record: no re-read
      w.pend = rev ? nullptr : t.slots + (uint64_t)w.x * B + s;
      c.held = victim;
      w.x = xn;
      w.v = vn;
      w.s = -1;
      w.tries = 0;
      c.viewed++;
      again = false;
    }
  }
  if (again) {  // the bin changed since its view
    if (++w.tries == 4) return ST_CONFLICT;
    load_view_fast<B>(t, w.x, w.v);
    c.viewed++;
    c.reviews++;
  }
  return WALK;
}

// Entries first .. first + 3 of the plan (those below n; the others repeat
// the last), loaded together.
__device__ __forceinline__ void load_entries(const Ctx& c, int first, int n, ulonglong2 (&e)[4]) {
#pragma unroll
  for (int u = 0; u < 4; u++) {
    const int i = min(first + u, n - 1);
    if (i < REG_ENTRIES) e[u] = make_ulonglong2(c.r0d, c.r0c);
    else e[u] = *reinterpret_cast<const ulonglong2*>(c.pe + 2 * i);
  }
}

// The writes of a chain, last slot first, then the releases (as commit,
// ck_insert.cuh).  An entry's content is the record its slot receives.  The
// last record of a two-choice walk is in its free slot already; rattle-kicking
// claims that slot, because its counter is in the metadata word, and takes it
// here (false if it was taken meanwhile, with nothing written).
template <int B, int POL>
__device__ __forceinline__ bool walk_commit(const DevTable& t, Ctx& c) {
  const int n = c.pn;
  if (n == 0) return true;
  ulonglong2 e[4];
  for (int first = (n - 1) & ~3; first >= 0; first -= 4) {
    load_entries(c, first, n, e);
#pragma unroll
    for (int u = 3; u >= 0; u--) {
      if (first + u >= n || e_sup(e[u].x)) continue;  // a later revisit of the slot writes it
      if (POL == P_RATTLE && first + u == n - 1) {
        if (!cas_slot(slot_at<B>(t, e[u].x), EMPTY, e[u].y)) return false;
        continue;
      }
      if (t.ordered_writes) fence_release();          // the copy lands before its source is overwritten
      st_slot(slot_at<B>(t, e[u].x), e[u].y);
    }
  }
  // nothing moved when a new key took a free slot: no order to keep
  if (POL != P_RATTLE || n > 1) fence_release();
  for (int first = 0; first < n; first += 4) {
    load_entries(c, first, n, e);
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (first + u >= n) continue;
      uint32_t delta = VER_ONE - (e_rev(e[u].x) ? 0u : 1u << e_slot(e[u].x));
      if (B == 1) delta += (e_new_r(e[u].x) - e_old_r(e[u].x)) << RATTLE_SHIFT;
      red_relaxed(t.meta + e_bin(e[u].x), delta);
    }
  }
  return true;
}

// The lanes whose walk ended, or that wait for a key, are served once they
// are WAITERS times the lanes still walking.  Measured, fill of 2^24 x 4 to
// 0.95 with queue-kicking (each against the next, same GPU): served as soon
// as one lane waits 7.80 ms, from 1/8, 1/4 and 1/2 of the walking lanes on
// 7.59, 7.37 and 7.16 (commits loading one entry at a time: 6.86 for 1/2 with
// four at a time), from as many on 6.44, from twice as many on 6.33.
//
// 80 registers (3 blocks of 256 threads on an SM; 4-slot queue-kicking spills
// nothing): 6.43 ms against 6.61 at 64, which spill.  One block waits for the launch before, which is
// enough to keep this one from completing first: blocks that are done make
// room for the next launch's (6.43 against 6.46 with every block waiting).
constexpr int WAITERS = 2;

// Searches that keep their first groups in shared memory (Search).  Measured,
// 4,194,304 x 4 to 0.95 / 1,500,007 x 8 to 0.97, against all of it in the
// region: sorted search 5.14 / 3.24 ms against 5.46 / 3.44, the hybrid 6.38 /
// 3.19 against 6.71 / 3.42; but BFS 6.24 / 3.15 against 6.02 / 3.16, and with
// ghosts sorted search 6.43 against 5.98 (4 slots), BFS 4.86 against 4.70 (8
// slots).  8 or 20 groups instead of 12 are slower.
template <int B, int POL, bool GHOST>
constexpr bool search_near = B > 1 && !GHOST && (POL == P_SORTED || POL == P_HYBRID);

// What a lane keeps of its insertion between two steps, and the steps: the
// walks above for two-choice tables without ghosts and for rattle-kicking,
// else the steps that the serial replay runs (ck_insert.cuh, ck_search.cuh).
template <int B, int POL, bool GHOST>
struct Lane {
  static constexpr bool SEARCH = is_search_policy<POL>;
  static constexpr bool NEAR = search_near<B, POL, GHOST>;
  static constexpr bool OWN = POL == P_RATTLE || (B > 1 && !GHOST && !SEARCH);
  using Dary = typename Choose<SEARCH, DarySearch, DaryKicks>::type;
  using Two = typename Choose<SEARCH, Search<B, NEAR>, Kicks<B>>::type;
  using Rest = typename Choose<B == 1, Dary, Two>::type;
  using State = typename Choose<OWN, Walk<B>, Rest>::type;

  static __device__ __forceinline__ int begin(const DevTable& t, Ctx& c, State& w, uint8_t* region) {
    if constexpr (SEARCH) {
      if (!region) return ST_ABORTED;
      if constexpr (B == 1) return search_first_dary<POL, true>(t, c, w, region);
      else return search_first<B, POL, GHOST, NEAR, true>(t, c, w, region);
    } else if constexpr (OWN) {
      return walk_begin<B, POL>(t, c, w);
    } else if constexpr (B == 1) {
      return random_dary_first(t, c, w);
    } else if constexpr (POL == P_QUEUE) {
      return queue_first<B, GHOST>(t, c, w);
    } else {
      return random_first<B, GHOST>(t, c, w);
    }
  }
  static __device__ __forceinline__ int step(const DevTable& t, Ctx& c, State& w) {
    if constexpr (SEARCH) {
      if constexpr (B == 1) return search_rounds_dary<POL, true>(t, c, w);
      else return search_rounds<B, POL, GHOST, NEAR, true>(t, c, w);
    } else if constexpr (OWN) {
      return walk_step<B, POL>(t, c, w);
    } else if constexpr (B == 1) {
      return random_dary_kick(t, c, w);
    } else if constexpr (POL == P_QUEUE) {
      return queue_kick<B, GHOST>(t, c, w);
    } else {
      return random_kick<B, GHOST>(t, c, w);
    }
  }
  static __device__ __forceinline__ bool finish(const DevTable& t, Ctx& c) {
    if constexpr (OWN) return walk_commit<B, POL>(t, c);
    else return commit<B>(t, c);
  }
};

// Insert the keys of `src`, by a whole warp; region: the lane's search region.  `src` gives each lane its keys
// and the table they go into, and counts what became of them:
//   more            keys may be left (the same in all lanes)
//   take(idle)      the whole warp calls; true in a lane of `idle` that got a
//                   key (src.key, src.val)
//   table()         the lane's table
//   done(over, c, st, aborts)   the whole warp calls: the ends of the keys of
//                   the lanes with `over`
template <int B, int POL, bool GHOST, class Src>
__device__ __forceinline__ void walk_keys(Src& src, uint64_t* local_e, uint8_t* region = nullptr) {
  using L = Lane<B, POL, GHOST>;
  constexpr bool SEARCH = L::SEARCH;
  // a lane has no key; has one whose next attempt begins; walks; has an
  // attempt that ended with st; waits, before its next attempt or for a
  // scratch plan (searches)
  enum Mode { IDLE, READY, WALKING, ENDED, WAITING };
  constexpr int WANT_BIG = -2;
  int mode = IDLE, st = ST_OK;
  Ctx c;
  c.ghosts_made = c.dup_evict = 0;
  c.kicks = c.viewed = c.viewed0 = c.reviews = 0;
  typename L::State w;
  uint32_t fails = 0, aborts = 0, wake = 0;
  for (;;) {
    if (mode == WAITING && (int)((uint32_t)clock() - wake) >= 0) {
      mode = READY;
      // A search that ran out of budget (WANT_BIG), or whose path outgrew its
      // plan, asks the pool for a scratch plan and waits for the next time to
      // ask beside the other lanes, among them holders of plans (polling in
      // place held all of them up: BFS, 2^22 x 4 filled to 0.982, 4.3 s and
      // 56,200 keys FAILED against 2.2 s and 38,900).  It asks for about as long as
      // acquire_long polls and then goes on without.  A negative long_id or
      // big_id counts the times.
      if (SEARCH && (st == ST_LONG || c.big_id <= WANT_BIG)) {
        const DevTable& t = src.table();
        const bool plan = st == ST_LONG;
        int id = plan ? c.long_id : c.big_id;
        const int got = try_long(t, fmix32(c.key - (uint32_t)id));
        if (got >= 0) {
          id = got;
          if (plan) use_plan(t, c, got);
          else clear_big_space(t.long_scratch + (uint64_t)got * LONG_REGION);
        } else if (id > -(int)(256 + 40 * t.n_long)) {
          id--;
          wake = (uint32_t)clock() + 2 * backoff_ns(5, c.key - (uint32_t)id);
          mode = WAITING;
        } else {
          id = -1;
          if (plan) {
            st = ST_ABORTED;
            mode = ENDED;
          }
        }
        if (plan) c.long_id = id;
        else c.big_id = id;
      }
    }
    const unsigned walking = __ballot_sync(0xFFFFFFFFu, mode == WALKING);
    const unsigned waiting = __ballot_sync(0xFFFFFFFFu, mode == WAITING);
    const unsigned need = __ballot_sync(0xFFFFFFFFu, mode == ENDED || mode == READY || (mode == IDLE && src.more));
    if (!(walking | waiting | need)) break;
    if (need && __popc(need) >= WAITERS * __popc(walking)) {
      bool over = false;
      if (mode == ENDED) {  // as insert_one ends an attempt
        bool undone = false;
        if (st == ST_OK) {
          over = L::finish(src.table(), c);
          if (!over) st = ST_CONFLICT;
          undone = !over;
        }
        if (!over) {
          release_all(src.table(), c, undone);
          const bool ran_out = st == ST_FAILED || c.capped;
          const bool longer = SEARCH && st == ST_LONG;  // the path goes on in a scratch plan
          if (longer) {
            over = c.long_id >= 0;
            if (over) st = ST_FAILED;
            wake = (uint32_t)clock();
            mode = WAITING;
          } else if (SEARCH && st == ST_ABORTED) {  // no search region
            over = true;
          } else if (ran_out) {
            over = ++fails > (st == ST_FAILED ? 6u : 32u);
            if (over) st = ST_FAILED;
            // a search out of budget tries again in a larger space
            if (SEARCH && !over && c.big_id < 0) c.big_id = WANT_BIG;
          } else {
            aborts++;
          }
          if (!over && !longer && ++c.attempt >= src.table().max_retries) {
            st = ST_ABORTED;
            over = true;
          }
          if (!over && !longer) {
            wake = (uint32_t)clock() + 2 * backoff_ns(ran_out ? 6 + 2 * fails : c.attempt, c.key);
            mode = WAITING;
          }
        }
      }
      if (over && c.long_id >= 0) release_long(src.table(), c.long_id);
      if (SEARCH && over && c.big_id >= 0) release_long(src.table(), c.big_id);
      if (__any_sync(0xFFFFFFFFu, over)) src.done(over, c, st, aborts);
      if (over) mode = IDLE;
      // keys for the idle lanes
      const unsigned idle = __ballot_sync(0xFFFFFFFFu, mode == IDLE);
      if (idle && src.more && src.take(idle)) {
        c.key = src.key;
        c.krec = ((uint64_t)src.key << 32) | src.val;
        c.attempt = 0;
        c.viewed = 0;
        c.reviews = 0;
        c.long_id = -1;
        c.big_id = -1;
        fails = 0;
        aborts = 0;
        mode = READY;
      }
      if (mode == READY) {
        c.kicks = 0;
        c.draws = 0;
        c.viewed0 = c.viewed;
        c.foreign = 0;
        c.capped = 0;
        c.ghosts_made = 0;
        c.dup_evict = 0;
        if (c.long_id < 0) {
          c.pe = local_e;
          c.pcap = MAX_CHAIN;
        }
        c.pn = 0;
        st = L::begin(src.table(), c, w, region);
        mode = st == WALK ? WALKING : ENDED;
      }
    }
    if (mode == WALKING) {
      st = L::step(src.table(), c, w);
      if (st != WALK) mode = ENDED;
    } else if (!walking && !need) {
      __nanosleep(100);
    }
    __syncwarp();
  }
}

// The keys lo .. hi - 1 of a batch, into one table.
template <int B, int POL, bool LOOK>
struct BatchKeys {
  const DevTable& t;
  const uint32_t *keys, *vals;
  uint8_t* status;
  uint32_t* viewed_out;
  uint64_t hi, load_base;
  BlockTally& bt;
  LookState& ls;
  bool more;
  uint64_t i;
  uint32_t key, val;

  __device__ __forceinline__ const DevTable& table() const { return t; }
  __device__ __forceinline__ bool take(unsigned idle) {
    uint64_t got = hi;
    if constexpr (!LOOK) {  // straight from the block's range
      const uint32_t lane = lane_id();
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(&ls.next, (unsigned long long)__popc(idle));
      base = __shfl_sync(0xFFFFFFFFu, base, 0);
      more = base + __popc(idle) < hi;
      if ((idle >> lane) & 1u) got = base + __popc(idle & ((1u << lane) - 1));
    } else {
      more = ls.template take<B, POL>(t, keys, vals, status, viewed_out, hi, load_base, idle, bt, got);
    }
    if (got >= hi) return false;
    i = got;
    key = __ldcs(keys + i);
    val = __ldcs(vals + i);
    if (!LOOK && key == RESERVED_KEY) {
      if (status) status[i] = ST_INVALID;
      if (viewed_out) viewed_out[i] = 0;
      return false;
    }
    return true;
  }
  __device__ __forceinline__ void done(bool over, const Ctx& c, int st, uint32_t aborts) {
    if (over) {
      const uint32_t v = c.viewed - c.viewed0;
      if (status) status[i] = (uint8_t)st;
      if (viewed_out) viewed_out[i] = v;
      const uint32_t b = load_bucket(load_base + i, t.total_slots);
      atomicAdd(&bt.views[b], v);
      atomicAdd(&bt.cnt[b], 1u);
      if (st == ST_OK) atomicAdd(&bt.chain[chain_bucket(c.kicks)], 1u);
    }
    const KeySums s = sum_keys(over, c, st, aborts);
    if (lane_id() == 0) add_sums<true>(bt.bc, s);
    if (over && st == ST_OK) {
      if (c.ghosts_made) count_add(&bt.bc[C_GHOSTS_MADE], c.ghosts_made);
      if (c.dup_evict) count_add(&bt.bc[C_DUP_EVICT], c.dup_evict);
    }
  }
};

// Blocks of 256 threads on an SM.  Fewer searches at a time leave more of L2
// to the table: 8-slot sorted search 3.44 ms with 2 blocks, 3.54 with 3.
template <int B, int POL, bool GHOST>
constexpr int walk_blocks_per_sm =
    B == 1 ? 4 : is_search_policy<POL> && (B == 8 || search_near<B, POL, GHOST>) ? 2 : 3;

// dynamic shared memory of a block
template <int B, int POL, bool GHOST>
constexpr size_t walk_shared(uint32_t block) { return search_near<B, POL, GHOST> ? (size_t)block * NEAR_BYTES : 0; }

// Consecutive launches may overlap (programmatic dependent launch): each block
// lets the next launch start at once (a search once it has its slabs), and
// block 0 ends after the launch before (see WAITERS), so a launch completes only after its predecessor.
// Insertions of distinct absent keys commute under the claim protocol, so the
// overlap changes no result.
template <int B, int POL, bool GHOST>
__global__ void __launch_bounds__(256, walk_blocks_per_sm<B, POL, GHOST>) k_insert_walk(DevTable t, const uint32_t* __restrict__ keys,
                                                        const uint32_t* __restrict__ vals, uint64_t n,
                                                        uint8_t* __restrict__ status,
                                                        uint32_t* __restrict__ viewed_out, uint64_t load_base) {
  constexpr bool SEARCH = is_search_policy<POL>;
  if (!SEARCH) asm volatile("griddepcontrol.launch_dependents;");
  __shared__ BlockTally bt;
  __shared__ LookState ls;
  const uint64_t per = (n + gridDim.x - 1) / gridDim.x;
  const uint64_t lo = min(n, (uint64_t)blockIdx.x * per), hi = min(n, lo + per);
  __shared__ int s_slab[SEARCH ? SLABS_PER_BLOCK : 1];
  bt.clear();
  ls.begin(t, lo, load_base);
  if (SEARCH && threadIdx.x < 32) {
    const bool got = take_slabs(t, s_slab, (int)((blockDim.x + SLAB - 1) / SLAB));
    if (!got && threadIdx.x == 0) s_slab[0] = -1;
  }
  __syncthreads();
  if (SEARCH) asm volatile("griddepcontrol.launch_dependents;");  // see take_slabs
  PlanStore<MAX_CHAIN> store;
  BatchKeys<B, POL, (B > 1 && !GHOST)> src{t, keys, vals, status, viewed_out, hi, load_base, bt, ls, true, 0, 0, 0};
  walk_keys<B, POL, GHOST>(src, store.e, SEARCH ? slab_region(t, s_slab) : nullptr);
  __syncthreads();
  bt.flush(t);
  if (SEARCH && threadIdx.x == 0) release_slabs(t, s_slab);
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");  // see WAITERS
}

}  // namespace ck
