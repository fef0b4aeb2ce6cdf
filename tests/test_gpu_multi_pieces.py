"""The batched insertion's pieces: tables smaller and larger than a piece of
512 keys, sizes just around it, 4- and 8-slot tables in any order or only one
kind, tables with no keys, keys past a tile's end, and reserved keys.  Every
table ends with its own keys and counts them in its own counters."""
import numpy as np
import pytest
import torch

from paper_1605_05236_gb300 import ck, inputs
from paper_1605_05236_gb300.multi import MULTI_BLOCK, MULTI_TILE, MultiTable

pytestmark = pytest.mark.gpu

SHAPES = {
    "edges": ([256] * 6, [4, 8, 4, 8, 4, 4], [511, 512, 513, 1025, 1, 0]),
    "only-8": ([300, 5, 4001], [8, 8, 8], [2000, 0, 31000]),
    "only-4": ([2, 77, 10007], [4, 4, 4], [7, 290, 38000]),
    "one": ([65536], [4], [249000]),
    "many": (list(range(40, 340)), [4 + 4 * (i % 3 == 0) for i in range(300)],
             [int(0.93 * b * (4 + 4 * (i % 3 == 0))) for i, b in enumerate(range(40, 340))]),
}


@pytest.mark.parametrize("policy", [ck.QUEUE, ck.RANDOM, ck.QUEUE | ck.GHOST])
@pytest.mark.parametrize("tile,block", [(256, 64), (4096, 128), (1 << 16, 256)])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_every_table_holds_its_keys(shape, tile, block, policy):
    bins, slots, n_keys = SHAPES[shape]
    m = MultiTable(bins, slots, n_keys, policy, seed=9)
    m.set_param(MULTI_TILE, tile)
    m.set_param(MULTI_BLOCK, block)
    total = int(sum(n_keys))
    keys, _ = inputs.distinct_keys(total, 31)
    sent = keys.copy()
    sent[5::101] = 0xFFFFFFFF
    vals = inputs.values_for(sent)
    st = torch.full((total,), 99, dtype=torch.uint8, device="cuda")
    m.insert(ck.as_u32_tensor(sent), ck.as_u32_tensor(vals), st)
    want = np.where(sent == 0xFFFFFFFF, ck.ST_INVALID, 0).astype(np.uint8)
    assert np.array_equal(st.cpu().numpy(), want)
    for i in range(len(bins)):
        a = int(m.offsets[i])
        k = sent[a:a + n_keys[i]]
        k = k[k != 0xFFFFFFFF]
        assert m.contents(i) == dict(zip(k.tolist(), inputs.values_for(k).tolist()))
        s = m.stats(i)
        assert s["inserts_ok"] == s["size"] == len(k)
        assert s["bins_viewed_all"] >= s["bins_viewed"] >= len(k)
    m.clear()
    assert m.stats()["size"] == 0 and all(m.contents(i) == {} for i in range(min(3, len(bins))))
