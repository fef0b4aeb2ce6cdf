"""Calls queued back to back on one stream without a synchronisation between
them: an upsert finds the keys of the insert and of the upsert before it
(overwritten in place, one copy a key), an insert after an upsert changes
nothing of it, and a serial replay runs alone between concurrent inserts."""
import numpy as np
import pytest
import torch

import oracle
from paper_1605_05236_gb300 import ck, inputs
from table_checks import check_table

pytestmark = pytest.mark.gpu

SHAPES = [(1 << 18, 4, 2, ck.QUEUE, 0.93), (1 << 16, 8, 2, ck.SORTED, 0.93), (1 << 16, 8, 2, ck.QUEUE | ck.GHOST, 0.9),
          (1 << 18, 4, 2, ck.RANDOM, 0.9), (1 << 18, 1, 4, ck.BFS, 0.9), (1 << 18, 1, 4, ck.RATTLE, 0.9)]


@pytest.mark.parametrize("bins,B,d,policy,load", SHAPES)
def test_upserts_see_the_calls_before_them(bins, B, d, policy, load):
    n = inputs.load_target(bins * B, load)
    m = n // 16
    keys, _ = inputs.distinct_keys(n, 41)
    kt = ck.as_u32_tensor(keys)
    vals = [ck.as_u32_tensor((inputs.values_for(keys) + np.uint32(i)).astype(np.uint32)) for i in range(4)]
    st = [torch.full((n,), 99, dtype=torch.uint8, device="cuda") for _ in range(5)]
    t = ck.CuckooTable(bins, B, d, policy, seed=6)
    t.insert(kt[:n - m], vals[0][:n - m], st[0][:n - m])                           # insert
    t.insert(kt[:n - m], vals[1][:n - m], st[1][:n - m], upsert=True)              # the same keys: all present
    t.insert(kt[:m], vals[2][:m], st[2][:m], upsert=True)                          # a small call, then one beside it
    t.insert(kt[:m], vals[3][:m], st[3][:m], upsert=True)
    t.insert(kt[n - m:], vals[0][n - m:], st[4][:m])                               # other keys, inserted
    s = t.stats()
    got = [x.cpu().numpy() for x in st]
    assert (got[0][:n - m] == ck.ST_OK).all() and (got[4][:m] == ck.ST_OK).all()
    assert (got[1][:n - m] == ck.ST_UPDATED).all(), np.bincount(got[1][:n - m])
    assert (got[2][:m] == ck.ST_UPDATED).all() and (got[3][:m] == ck.ST_UPDATED).all()
    assert s["size"] == n and s["updates"] == n - m + 2 * m and s["inserts_ok"] == n
    slots, meta = t.export()
    assert check_table(slots, meta, bins, B, d)["size"] == n  # one copy a key (two of a ghost pair)
    v, f = t.lookup(kt)
    want = np.concatenate([ck.u32_numpy(vals[3][:m]), ck.u32_numpy(vals[1][m:n - m]), ck.u32_numpy(vals[0][n - m:])])
    assert bool((f == 1).all()) and np.array_equal(ck.u32_numpy(v), want)


@pytest.mark.parametrize("bins,B,policy", [(1 << 10, 4, ck.QUEUE), (1 << 10, 4, ck.SORTED)])
def test_a_serial_replay_runs_alone(bins, B, policy):
    n = inputs.load_target(bins * B, 0.95)
    keys, _ = inputs.distinct_keys(n, 43)
    vals = inputs.values_for(keys)
    ref = oracle.OracleTable(bins, B, 2, policy, rng_seed=7, cap=500)
    cut = n * 3 // 4
    ost, oviewed, _ = ref.insert(keys[:cut], vals[:cut], trace=True)
    kt, vt = ck.as_u32_tensor(keys), ck.as_u32_tensor(vals)
    t = ck.CuckooTable(bins, B, 2, policy, seed=7)
    viewed = torch.zeros(cut, dtype=torch.int32, device="cuda")
    st = t.insert(kt[:cut], vt[:cut], viewed=viewed, serial=True)
    rest = t.insert(kt[cut:], vt[cut:])
    assert np.array_equal(st.cpu().numpy(), ost) and np.array_equal(ck.u32_numpy(viewed), oviewed)
    assert (rest.cpu().numpy() == ck.ST_OK).all()
    assert t.contents() == dict(zip(keys.tolist(), vals.tolist()))
