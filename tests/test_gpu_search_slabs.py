"""Search tables whose launches overlap share one pool of search regions: a call
that follows one with many keys that end FAILED (their bins are full, and so
are all bins the searches can reach) waits for the regions that call holds,
however long, and places every key that has room."""
import numpy as np
import pytest
import torch

from paper_1605_05236_gb300 import ck, inputs
from table_checks import bins_np, check_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d,policy,warp", [(4, 2, ck.BFS | ck.GHOST, 0), (8, 2, ck.SORTED | ck.GHOST, 0),
                                             (4, 2, ck.BFS, 1), (1, 3, ck.BFS, 0), (1, 4, ck.SORTED, 0)])
def test_calls_behind_failing_searches_place_their_keys(B, d, policy, warp):
    bins, small = 1024, {2: 128, 3: 256, 4: 384}[d]
    keys, _ = inputs.distinct_keys(4_000_000, 29)
    kb = bins_np(keys, bins, d)
    inside = keys[(kb < small).all(axis=1)][:small * B + 50_000]  # a closed set of bins, far too many keys
    outside = keys[(kb >= small).all(axis=1)]
    m = (bins - small) * B // 6
    t = ck.CuckooTable(bins, B, d, policy, seed=2)
    if warp:
        t.set_param(ck.PARAM_SEARCH_WARP, 1)
    calls = [inside] + [outside[i * m:(i + 1) * m] for i in range(3)]
    dev = [(ck.as_u32_tensor(k), ck.as_u32_tensor(inputs.values_for(k)),
            torch.full((len(k),), 99, dtype=torch.uint8, device="cuda")) for k in calls]
    torch.cuda.synchronize()
    for k, v, st in dev:
        t.insert(k, v, st)
    first, *rest = [st.cpu().numpy() for _, _, st in dev]
    for st in rest:
        assert (st == ck.ST_OK).all(), np.bincount(st)
    assert (first == ck.ST_OK).sum() <= small * B
    assert (first != ck.ST_INVALID).all() and (first != 99).all()
    slots, meta = t.export()
    assert check_table(slots, meta, bins, B, d)["size"] == int((first == ck.ST_OK).sum()) + 3 * m
    t.close()
