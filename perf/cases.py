"""The calls a user of this library makes, as cases to be timed.

listed() names the cases, draw(rng) gives one more of the same ranges;
prepare(case, seed) makes what a program holds before the call (tables, key
and result buffers, traces), run(state) is one pass through the public entry
points, exact(case, seed) is what that pass returns, from the definition of
the operations alone, and work(case) the bytes a pass cannot do without.

Kinds of pass:
  point   a few hundred keys upserted, looked up and deleted in a resident
          table: the smallest calls
  build   a table filled from empty in batches, then probed (the build and
          probe side of a join, or an index rebuilt)
  lookup  one bulk lookup in a resident table
  churn   resident keys deleted (with requests for some that are gone) and
          inserted again in a table that stays near its load, then probed: a
          cache or an index under turnover
  multi   many independent tables of uneven sizes filled by one launch, then
          probed
  serve   a trace of lookup, insert and delete requests from host memory
          through the request loop, and the trace that undoes its writes
  txn     transactions of inserts, reads, overwrites and deletes on many
          trial tables
Every pass leaves its table holding the keys it held before (or starts by
clearing it), so a pass can be repeated.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_1605_05236_gb300 import ck, inputs
from paper_1605_05236_gb300.multi import MultiTable
from paper_1605_05236_gb300.serve import OP_DELETE, OP_INSERT, OP_LOOKUP, Server
from paper_1605_05236_gb300.txn import CLAIM, LOCAL_RETRY, SYSTEM, TxnTable

M32 = 0xFFFFFFFF
VALUE_MUL = 2654435761  # value of a key: key * VALUE_MUL mod 2^32
CHUNK = 1 << 25


def listed():
    return [
        # the smallest calls: an application keeps an index resident and
        # touches 512 keys at a time, half of them new
        {"name": "point_512", "kind": "point", "bins": 1 << 20, "B": 4, "policy": "queue", "load": 0.93, "n": 256},
        # one small table that stays in L2: all keys in one call, as many
        # probes as there are slots
        {"name": "build_small_random", "kind": "build", "bins": 1 << 14, "B": 4, "d": 2, "policy": "random",
         "ghost": False, "load": 0.95, "batch": 1 << 20, "probes": 65536},
        # the benchmark's fill: 512 MiB of 4-slot bins to 0.95 in batches of
        # 2^20 keys as they arrive, and the first probe batch
        {"name": "build_queue_4slot", "kind": "build", "bins": 1 << 24, "B": 4, "d": 2, "policy": "queue",
         "ghost": False, "load": 0.95, "batch": 1 << 20, "probes": 1 << 22},
        # a search policy on 8-slot bins, no power of two anywhere: the
        # densest tables
        {"name": "build_sorted_8slot", "kind": "build", "bins": 3000017, "B": 8, "d": 2, "policy": "sorted",
         "ghost": False, "load": 0.97, "batch": 1000003, "probes": 1000003},
        # ghost insertions: two copies of a key while there is room
        {"name": "build_ghost_4slot", "kind": "build", "bins": 1 << 22, "B": 4, "d": 2, "policy": "queue",
         "ghost": True, "load": 0.95, "batch": 1 << 19, "probes": 1 << 20},
        # single-slot bins with four choices, rattle-kicking
        {"name": "build_rattle_d4", "kind": "build", "bins": 1 << 24, "B": 1, "d": 4, "policy": "rattle",
         "ghost": False, "load": 0.94, "batch": 1 << 20, "probes": 1 << 22},
        # the benchmark's lookups: 2^26 keys, half of them absent
        {"name": "lookup_bulk_4slot", "kind": "lookup", "bins": 1 << 24, "B": 4, "d": 2, "policy": "queue",
         "load": 0.95, "n": 1 << 26, "hit": 0.5},
        # a mostly-hit lookup of odd size in 8-slot bins
        {"name": "lookup_8slot", "kind": "lookup", "bins": 5000011, "B": 8, "d": 2, "policy": "queue",
         "load": 0.97, "n": 20000003, "hit": 0.9},
        # turnover in a nearly full table: the benchmark's 2^22 deletes, and
        # as many insertions at that load
        {"name": "churn_4slot", "kind": "churn", "bins": 1 << 24, "B": 4, "policy": "queue", "load": 0.95,
         "n": 1 << 22, "batch": 1 << 20},
        # the batched form: 4096 tables, 2^10 .. 2^18 bins, replayed from a
        # captured graph
        {"name": "multi_4096", "kind": "multi", "tables": 4096, "lo": 10, "hi": 18, "load": 0.95, "graph": True,
         "probes": 1 << 22},
        # the serving form on a 2 GB table: requests of 1 .. 2^16 keys
        {"name": "serve_mixed", "kind": "serve", "bins": 1 << 26, "load": 0.95, "requests": 2048, "max_log2": 16,
         "lookup": 0.75, "insert": 0.20},
        # 100 trial tables of 2^12 x 8, 15 workers, transactions of 20
        # operations (an order or a payment), filled from empty to 0.89
        {"name": "txn_15_workers", "kind": "txn", "bins": 1 << 12, "trials": 100, "workers": 15, "txns": 290,
         "ops": 20, "mix": "1:0:1:1"},
    ]


# loads every key of a draw goes in at, by shape and policy: somewhat below
# where chains reach their cap
_TOP_LOAD = {(4, 2): 0.95, (8, 2): 0.97, (1, 3): 0.86, (1, 4): 0.93}


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _two_choice(rng):
    return rng.choice([4, 4, 8])


def draw(rng):
    kind = rng.choice(["point", "build", "build", "build", "build", "lookup", "lookup", "churn", "multi", "serve", "txn"])
    if kind == "point":
        return {"kind": kind, "bins": _log(rng, 1 << 12, 1 << 22), "B": _two_choice(rng),
                "policy": rng.choice(["queue", "random", "bfs"]), "load": round(rng.uniform(0.3, 0.94), 3),
                "n": _log(rng, 8, 4096)}
    if kind == "build":
        B, d = rng.choice([(4, 2), (4, 2), (8, 2), (8, 2), (1, 3), (1, 4)])
        top = _TOP_LOAD[(B, d)]
        if B == 1:
            policy, ghost = rng.choice(["rattle", "random", "sorted"]), False
        else:
            policy, ghost = rng.choice(["queue", "random", "bfs", "sorted", "hybrid"]), rng.random() < 0.3
        if B == 1 and policy == "sorted":
            top -= 0.04
        slots = _log(rng, 1 << 16, 1 << 25)
        return {"kind": kind, "bins": slots // B + rng.randrange(64), "B": B, "d": d, "policy": policy, "ghost": ghost,
                "load": round(rng.uniform(top - 0.35, top), 3), "batch": _log(rng, slots // 256, slots // 16),
                "probes": _log(rng, 1 << 12, 1 << 22)}
    if kind == "lookup":
        B, d = rng.choice([(4, 2), (8, 2), (1, 3), (1, 4)])
        return {"kind": kind, "bins": _log(rng, 1 << 14, 1 << 26) // B, "B": B, "d": d,
                "policy": "rattle" if B == 1 else "queue", "load": round(rng.uniform(0.5, _TOP_LOAD[(B, d)]), 3),
                "n": _log(rng, 1000, 1 << 26), "hit": round(rng.random(), 2)}
    if kind == "churn":
        slots = _log(rng, 1 << 18, 1 << 26)
        n = _log(rng, slots // 256, slots // 16)
        return {"kind": kind, "bins": slots // 4, "B": 4, "policy": rng.choice(["queue", "random"]),
                "load": round(rng.uniform(0.8, 0.95), 3), "n": n, "batch": _log(rng, max(1, n // 8), n)}
    if kind == "multi":
        lo = rng.randrange(8, 12)
        return {"kind": kind, "tables": _log(rng, 64, 2048), "lo": lo, "hi": lo + rng.randrange(2, 7),
                "load": round(rng.uniform(0.6, 0.95), 3), "graph": rng.random() < 0.5, "probes": _log(rng, 1 << 12, 1 << 22)}
    if kind == "serve":
        look = round(rng.uniform(0.4, 0.9), 2)
        return {"kind": kind, "bins": _log(rng, 1 << 21, 1 << 25), "load": round(rng.uniform(0.6, 0.94), 3),
                "requests": _log(rng, 64, 1024), "max_log2": rng.randrange(6, 14), "lookup": look,
                "insert": round((1 - look) * rng.uniform(0.4, 0.8), 3)}
    return {"kind": "txn", "bins": _log(rng, 1 << 12, 1 << 14), "trials": _log(rng, 50, 100),
            "workers": rng.randrange(10, 16), "txns": _log(rng, 30, 150), "ops": rng.randrange(5, 21),
            "mix": rng.choice(["1:0:1:1", "2:1:2:2"])}


# ---- inputs -----------------------------------------------------------


def _keys(seed, start, n):
    """n distinct keys (int32 bit patterns, never 0xFFFFFFFF): counters
    start .. start + n through a bijective 32-bit mixer (Wellons, "lowbias32"),
    so segments that do not share counters share no key.  Uses n + 1 counters."""
    base, twist = (seed * 0x9E3779B1 + 0x1234567) & M32, (seed * 0x85EBCA77 + 0xC2B2AE3D) & M32

    def mix(x):
        x = ((x + base) & M32) ^ twist
        x = x ^ (x >> 16)
        x = (x * 0x7FEB352D) & M32
        x = x ^ (x >> 15)
        x = (x * 0x846CA68B) & M32
        return (x ^ (x >> 16)).to(torch.int32)

    out = torch.empty(n, dtype=torch.int32, device="cuda")
    spare = mix(torch.tensor([start + n], dtype=torch.int64, device="cuda"))
    for a in range(0, n, CHUNK):
        b = min(n, a + CHUNK)
        k = mix(torch.arange(start + a, start + b, dtype=torch.int64, device="cuda"))
        out[a:b] = torch.where(k == -1, spare, k)
    return out


def _values(keys):
    out = torch.empty_like(keys)
    for a in range(0, keys.numel(), CHUNK):
        k = keys[a:a + CHUNK].to(torch.int64) & M32
        out[a:a + CHUNK] = ((k * VALUE_MUL) & M32).to(torch.int32)
    return out


def _sample(keys, n, gen):
    """n of the keys: distinct ones while there are enough."""
    if n <= keys.numel():
        return keys[torch.randperm(keys.numel(), generator=gen, device="cuda")[:n]]
    return keys[torch.randint(keys.numel(), (n,), generator=gen, device="cuda")]


def _probes(keys, seed, absent_start, n, hit):
    """n probe keys, n * hit of them present, in random order; and which."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n_hit = int(round(n * hit))
    p = torch.cat([_sample(keys, n_hit, gen), _keys(seed, absent_start, n - n_hit)])
    here = torch.zeros(n, dtype=torch.uint8, device="cuda")
    here[:n_hit] = 1
    order = torch.randperm(n, generator=gen, device="cuda")
    return p[order].contiguous(), here[order].contiguous()


def _found(probes, here):
    """What a lookup of the probes returns."""
    return _values(probes) * here.to(torch.int32), here


def _policy(case):
    return ck.POLICY_NAMES[case["policy"]] | (ck.GHOST if case.get("ghost") else 0)


def _table(case, seed):
    t = ck.CuckooTable(case["bins"], case["B"], case.get("d", 2), _policy(case), seed=seed)
    if case["B"] == 1:  # the hash family and the chain cap that single-slot tables are filled with
        t.set_param(ck.PARAM_HASH_FAMILY, 1)
        if case["policy"] == "random":
            t.set_param(ck.PARAM_CHAIN_CAP, 4096)
    return t


def _n_keys(case):
    return inputs.load_target(case["bins"] * case["B"], case["load"])


def _fill(t, keys, batch):
    vals = _values(keys)
    for a in range(0, keys.numel(), batch):
        t.insert_batch(keys[a:a + batch], vals[a:a + batch])


def _u8(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


def _i32(n):
    return torch.empty(n, dtype=torch.int32, device="cuda")


def _slices(n, batch):
    return [slice(a, min(n, a + batch)) for a in range(0, n, batch)]


# ---- what a pass works on ---------------------------------------------


def _point_keys(case, seed):
    n = case["n"]
    keys = _keys(seed, 0, _n_keys(case))
    new = _keys(seed, 1 << 30, n)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    both = torch.cat([_sample(keys, min(n, keys.numel()), gen), new])
    here = torch.cat([torch.ones(both.numel() - n, dtype=torch.uint8, device="cuda"),
                      torch.zeros(n, dtype=torch.uint8, device="cuda")])
    order = torch.randperm(both.numel(), generator=gen, device="cuda")
    return keys, both[order].contiguous(), here[order].contiguous(), new


def _build_keys(case, seed):
    keys = _keys(seed, 0, _n_keys(case))
    probes, here = _probes(keys, seed, 1 << 30, case["probes"], 0.5)
    return keys, probes, here


def _lookup_keys(case, seed):
    keys = _keys(seed, 0, _n_keys(case))
    probes, here = _probes(keys, seed, 1 << 30, case["n"], case["hit"])
    return keys, probes, here


def _churn_keys(case, seed):
    """The keys that leave and come back; the delete requests, one in eight
    of them for a key that is not there; and the probes that follow."""
    keys, n = _keys(seed, 0, _n_keys(case)), case["n"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = _sample(keys, n, gen).contiguous()
    gone, present = torch.cat([out, _keys(seed, 3 << 29, n // 8)]), _u8(n + n // 8)
    present[:n], present[n:] = 1, 0
    order = torch.randperm(gone.numel(), generator=gen, device="cuda")
    return keys, out, gone[order].contiguous(), present[order].contiguous(), *_probes(keys, seed, 1 << 30, n // 4, 0.5)


def _multi_shapes(case):
    bins, slots = inputs.multi_shapes(case["tables"], 7, case["lo"], case["hi"])
    n_keys = [inputs.load_target(int(b) * int(s), case["load"]) for b, s in zip(bins, slots)]
    return bins, slots, np.array(n_keys, dtype=np.uint64)


def _multi_keys(case, seed):
    _, _, n_keys = _multi_shapes(case)
    total, n = int(n_keys.sum()), case["probes"]
    keys = _keys(seed, 0, total)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    # half the probes ask the table that holds the key, half another one
    at = torch.randint(total, (n,), generator=gen, device="cuda")
    ends = torch.from_numpy(np.cumsum(n_keys).astype(np.int64)).cuda()
    tab = torch.searchsorted(ends, at, right=True)
    here = torch.randint(2, (n,), generator=gen, device="cuda")
    tab = torch.where(here == 1, tab, (tab + 1) % case["tables"])
    return keys, keys[at].contiguous(), tab.to(torch.int32), here.to(torch.uint8)


def _serve_traces(case, seed):
    """The trace and its inverse: the second deletes what the first inserted
    and inserts what it deleted.  Lookups ask for keys that neither writes, or
    that are never in the table."""
    n_req, rng = case["requests"], np.random.default_rng(11)  # sizes, kinds and arrivals are the case's, keys the seed's
    keys = _keys(seed, 0, inputs.load_target(case["bins"] * 4, case["load"]))
    sizes = np.floor(2.0 ** (case["max_log2"] * rng.random(n_req))).astype(np.uint64)
    kind = np.searchsorted([case["lookup"], case["lookup"] + case["insert"]], rng.random(n_req), side="right")
    arrive = np.cumsum(rng.exponential(50.0, n_req)).astype(np.int64)  # 20k requests a millisecond
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.uint64)
    counts = [int(sizes[kind == o].sum()) for o in range(3)]
    half = keys.numel() // 2
    gen = torch.Generator(device="cuda").manual_seed(seed)
    look, here = _probes(keys[:half], seed, 1 << 30, counts[0], 0.5)
    take = keys[half:][torch.randperm(keys.numel() - half, generator=gen, device="cuda")[:counts[2]]]
    pool = [look.cpu().numpy(), _keys(seed, 3 << 30, counts[1]).cpu().numpy(), take.cpu().numpy()]
    here = here.cpu().numpy()
    total = int(sizes.sum())
    k, expect = np.empty(total, dtype=np.int32), np.zeros(total, dtype=np.uint8)
    pos = [0, 0, 0]
    for i in range(n_req):
        o, a, n = int(kind[i]), int(off[i]), int(sizes[i])
        k[a:a + n] = pool[o][pos[o]:pos[o] + n]
        expect[a:a + n] = here[pos[o]:pos[o] + n] if o == 0 else (0 if o == 1 else 1)
        pos[o] += n
    k = k.view(np.uint32)
    vals = inputs.values_for(k)
    op = np.array([OP_LOOKUP, OP_INSERT, OP_DELETE], dtype=np.uint32)[kind]
    inverse = np.array([OP_LOOKUP, OP_DELETE, OP_INSERT], dtype=np.uint32)[kind]
    fwd = {"op": op, "n_keys": sizes, "key_off": off, "arrive_ns": arrive, "keys": k, "vals": vals}
    return keys, fwd, dict(fwd, op=inverse), kind, expect


def _txn_work(case, seed):
    mix = tuple(int(x) for x in case["mix"].split(":"))
    return inputs.txn_workload(case["workers"], case["txns"], case["ops"], mix, seed=1000 + seed)


def prepare(case, seed):
    s = {"kind": case["kind"]}
    kind = case["kind"]
    if kind == "point":
        keys, both, _, new = _point_keys(case, seed)
        s["t"] = _table(case, seed)
        _fill(s["t"], keys, max(1, keys.numel() // 8))
        s["both"], s["bvals"], s["new"] = both, _values(both), new
        s["status"], s["vals"], s["found"] = _u8(both.numel()), _i32(both.numel()), _u8(both.numel())
        s["gone"] = _u8(new.numel())
    elif kind == "build":
        s["keys"], s["probes"], _ = _build_keys(case, seed)
        s["kvals"] = _values(s["keys"])
        s["t"] = _table(case, seed)
        n = s["keys"].numel()
        s["status"], s["vals"], s["found"] = _u8(n), _i32(case["probes"]), _u8(case["probes"])
        s["batches"] = [(s["keys"][i], s["kvals"][i], s["status"][i]) for i in _slices(n, case["batch"])]
    elif kind == "lookup":
        keys, s["probes"], _ = _lookup_keys(case, seed)
        s["t"] = _table(case, seed)
        _fill(s["t"], keys, max(1, keys.numel() // 64))
        s["vals"], s["found"] = _i32(case["n"]), _u8(case["n"])
    elif kind == "churn":
        keys, out, gone, _, s["probes"], _ = _churn_keys(case, seed)
        s["t"] = _table(case, seed)
        _fill(s["t"], keys, max(1, keys.numel() // 64))
        vals = _values(out)
        s["gone"], s["status"] = _u8(gone.numel()), _u8(out.numel())
        s["vals"], s["found"] = _i32(s["probes"].numel()), _u8(s["probes"].numel())
        s["deletes"] = [(gone[i], s["gone"][i]) for i in _slices(gone.numel(), case["batch"])]
        s["batches"] = [(out[i], vals[i], s["status"][i]) for i in _slices(out.numel(), case["batch"])]
    elif kind == "multi":
        bins, slots, n_keys = _multi_shapes(case)
        s["keys"], s["probes"], s["tab"], _ = _multi_keys(case, seed)
        s["kvals"], s["status"] = _values(s["keys"]), _u8(s["keys"].numel())
        s["vals"], s["found"] = _i32(case["probes"]), _u8(case["probes"])
        s["m"] = MultiTable(bins, slots, n_keys, ck.QUEUE, seed=seed)
        s["graph"] = s["m"].capture(s["keys"], s["kvals"], s["status"], clear=True) if case["graph"] else None
    elif kind == "serve":
        keys, s["fwd"], s["back"], _, _ = _serve_traces(case, seed)
        t = ck.CuckooTable(case["bins"], 4, 2, ck.QUEUE, seed=seed)
        _fill(t, keys, max(1, keys.numel() // 64))
        s["server"] = Server(t)
    else:
        w = _txn_work(case, seed)
        s["x"] = TxnTable(case["bins"], 8, case["trials"], seed=seed)
        s["op"] = torch.from_numpy(w["op"]).cuda()
        s["key"], s["val"] = ck.as_u32_tensor(w["key"]), ck.as_u32_tensor(w["val"])
        s["shape"] = (case["workers"], case["txns"], case["ops"])
    torch.cuda.synchronize()
    return s


def run(s):
    kind = s["kind"]
    if kind == "point":
        t = s["t"]
        t.insert(s["both"], s["bvals"], s["status"], upsert=True)
        t.lookup(s["both"], s["vals"], s["found"])
        t.delete(s["new"], s["gone"])
        return s["status"], s["vals"], s["found"], s["gone"]
    if kind == "build":
        t = s["t"]
        t.clear()
        for keys, vals, status in s["batches"]:
            t.insert_batch(keys, vals, status)
        t.lookup(s["probes"], s["vals"], s["found"])
        return s["status"], s["vals"], s["found"]
    if kind == "lookup":
        s["t"].lookup(s["probes"], s["vals"], s["found"])
        return s["vals"], s["found"]
    if kind == "churn":
        t = s["t"]
        for keys, gone in s["deletes"]:
            t.delete(keys, gone)
        for keys, vals, status in s["batches"]:
            t.insert_batch(keys, vals, status)
        t.lookup(s["probes"], s["vals"], s["found"])
        return s["gone"], s["status"], s["vals"], s["found"]
    if kind == "multi":
        m = s["m"]
        if s["graph"] is not None:
            s["graph"].launch()
        else:
            m.clear()
            m.insert(s["keys"], s["kvals"], s["status"])
        m.lookup(s["tab"], s["probes"], s["vals"], s["found"])
        return s["status"], s["vals"], s["found"]
    if kind == "serve":
        v0, s0, _ = s["server"].replay(s["fwd"])
        v1, s1, _ = s["server"].replay(s["back"])
        return v0.view(np.int32), s0, v1.view(np.int32), s1
    s["x"].reset()
    out = s["x"].run(s["op"], s["key"], s["val"], *s["shape"], flags=LOCAL_RETRY | CLAIM | SYSTEM)
    return out["status"], out["value"]


# ---- what a pass returns, by definition --------------------------------


def exact(case, seed):
    kind = case["kind"]
    if kind == "point":
        _, both, here, new = _point_keys(case, seed)
        ones = torch.ones_like(here)
        return here * ck.ST_UPDATED, _values(both), ones, torch.ones(new.numel(), dtype=torch.uint8, device="cuda")
    if kind == "build":
        keys, probes, here = _build_keys(case, seed)
        return (torch.zeros(keys.numel(), dtype=torch.uint8, device="cuda"),) + _found(probes, here)
    if kind == "lookup":
        _, probes, here = _lookup_keys(case, seed)
        return _found(probes, here)
    if kind == "churn":
        _, out, _, present, probes, here = _churn_keys(case, seed)
        return (present, torch.zeros(out.numel(), dtype=torch.uint8, device="cuda")) + _found(probes, here)
    if kind == "multi":
        keys, probes, _, here = _multi_keys(case, seed)
        return (torch.zeros(keys.numel(), dtype=torch.uint8, device="cuda"),) + _found(probes, here)
    if kind == "serve":
        _, fwd, back, kind_of, expect = _serve_traces(case, seed)
        of_key = np.repeat(kind_of, fwd["n_keys"].astype(np.int64))
        look = of_key == 0
        vals = np.where(look & (expect == 1), fwd["vals"], 0).astype(np.uint32).view(np.int32)
        undone = np.where(look, expect, np.where(of_key == 1, 1, 0)).astype(np.uint8)
        return vals, expect, vals, undone
    w = _txn_work(case, seed)
    status, value, table = [], [], {}
    for o, k, v in zip(w["op"].tolist(), w["key"].tolist(), w["val"].tolist()):
        old = table.get(k)
        if o == inputs.TX_INSERT:
            table[k] = v
            status.append(0)
        else:
            status.append(0 if old is None else 1)
            if old is not None and o == inputs.TX_OVERWRITE:
                table[k] = v
            elif old is not None and o == inputs.TX_DELETE:
                del table[k]
        value.append(old if o == inputs.TX_READ and old is not None else 0)
    status, value = np.array(status, dtype=np.uint8), np.array(value, dtype=np.uint32).view(np.int32)
    return (torch.from_numpy(np.tile(status, case["trials"])).cuda(),
            torch.from_numpy(np.tile(value, case["trials"])).cuda())


# ---- the least a pass moves ---------------------------------------------


def _probe_bytes(n, bin_bytes, table_bytes, hit, d=2):
    """Keys in, values and flags out, and the bins: all d of an absent key,
    (d + 1) / 2 of a present one on average, no bin more than once."""
    return n * 9 + min(table_bytes, n * bin_bytes * (d * (1 - hit) + (d + 1) / 2 * hit))


def work(case):
    kind = case["kind"]
    if kind == "multi":
        bins, slots, n_keys = _multi_shapes(case)
        table, n = int((bins * slots * 8).sum()), int(n_keys.sum())
        b = table + n * 9 + _probe_bytes(case["probes"], 48, table, 0.5) + case["probes"] * 4
    elif kind == "txn":
        n = case["workers"] * case["txns"] * case["ops"]
        b = n * 9 + case["trials"] * (n * 5 + case["bins"] * 64)
    elif kind == "serve":
        keys = case["requests"] * (2.0 ** case["max_log2"] - 1) / (case["max_log2"] * np.log(2.0))  # mean of log-uniform sizes
        b = 2 * keys * (case["lookup"] * (9 + 32 * 1.75) + (1 - case["lookup"]) * (9 + 32 * 2))
    else:
        bin_bytes, d = case["B"] * 8, case.get("d", 2)
        table = case["bins"] * bin_bytes
        if kind == "point":
            n = 2 * case["n"]
            b = n * 9 + _probe_bytes(n, bin_bytes, table, 1.0) + case["n"] * (5 + bin_bytes)
        elif kind == "build":
            b = table + _n_keys(case) * 9 + _probe_bytes(case["probes"], bin_bytes, table, 0.5, d)
        elif kind == "lookup":
            b = _probe_bytes(case["n"], bin_bytes, table, case["hit"], d)
        else:
            n = case["n"]
            b = n * (5 + 2 * bin_bytes + 9 + 2 * bin_bytes) + n // 8 * (5 + 2 * bin_bytes)
            b += _probe_bytes(n // 4, bin_bytes, table, 0.5)
    return {"bytes": int(b), "flops": 0}
