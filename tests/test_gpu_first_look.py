"""The concurrent insert kernels that take their keys through a first look,
32 a warp, and insert what found no room lane by lane (walks) or 32 at a
time (searches): batch sizes around a warp and a block, reserved keys in the
batch, statuses and bins viewed wanted or not, few insertions in flight, and
a fill to the loads where walks are long.  Every key gets the status and the
value the oracle's table gives it."""
import numpy as np
import pytest
import torch

import oracle
from paper_1605_05236_gb300 import ck, inputs
from table_checks import check_table

pytestmark = pytest.mark.gpu

POLICIES = [ck.QUEUE, ck.RANDOM, ck.BFS, ck.SORTED]


@pytest.mark.parametrize("policy", POLICIES)
@pytest.mark.parametrize("n", [1, 31, 32, 33, 127, 128, 129, 255, 257, 1000])
def test_batch_sizes_and_reserved_keys(policy, n):
    t = ck.CuckooTable(1 << 8, 4 if n % 2 else 8, 2, policy, seed=3)
    keys, _ = inputs.distinct_keys(n, 5)
    bad = np.arange(0, n, 7) if n > 1 else np.array([], dtype=int)
    sent = keys.copy()
    sent[bad] = 0xFFFFFFFF
    if n > t.total_slots * 0.9:
        sent = sent[:int(t.total_slots * 0.9)]
        bad = bad[bad < len(sent)]
    viewed = torch.full((len(sent),), 99, dtype=torch.int32, device="cuda")
    st = t.insert(ck.as_u32_tensor(sent), ck.as_u32_tensor(inputs.values_for(sent)), viewed=viewed)
    want = np.zeros(len(sent), dtype=np.uint8)
    want[bad] = ck.ST_INVALID
    assert np.array_equal(st.cpu().numpy(), want)
    v = viewed.cpu().numpy()
    assert (v[bad] == 0).all() and (v[want == 0] >= 1).all()
    good = sent[want == 0]
    assert t.contents() == dict(zip(good.tolist(), inputs.values_for(good).tolist()))
    s = t.stats()
    assert s["inserts_ok"] == s["size"] == len(good)
    views, counts = t.load_histogram()
    assert counts.sum() == len(good) and views.sum() == s["bins_viewed"] == int(v.sum())
    assert t.chain_histogram().sum() == len(good)


@pytest.mark.parametrize("inflight,ordered", [(0, 0), (0, 1), (32, 0), (4096, 0)])
@pytest.mark.parametrize("bins,B,policy,load", [(1 << 12, 4, ck.QUEUE, 0.95), (3001, 8, ck.QUEUE, 0.98),
                                                (1 << 12, 4, ck.RANDOM, 0.95), (3001, 8, ck.RANDOM, 0.97),
                                                (3001, 8, ck.SORTED, 0.97)])
def test_fill_holds_the_oracles_map(bins, B, policy, load, inflight, ordered):
    n = inputs.load_target(bins * B, load)
    keys, _ = inputs.distinct_keys(n, 23)
    vals = inputs.values_for(keys)
    ref = oracle.OracleTable(bins, B, 2, policy, rng_seed=7, cap=500)
    assert (ref.insert(keys, vals) == 0).all()
    t = ck.CuckooTable(bins, B, 2, policy, seed=7)
    t.set_param(ck.PARAM_MAX_INFLIGHT, inflight)
    t.set_param(ck.PARAM_ORDERED_WRITES, ordered)
    kt, vt = ck.as_u32_tensor(keys), ck.as_u32_tensor(vals)
    for a in range(0, n, 1777):  # statuses not wanted
        t.insert_batch(kt[a:a + 1777], vt[a:a + 1777])
    assert t.contents() == ref.contents()
    slots, meta = t.export()
    assert check_table(slots, meta, bins, B, 2)["size"] == n
