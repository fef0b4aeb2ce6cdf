"""The batched insertion with tiles far larger than its tables: the pieces it
hands out follow the keys there are, not the tile size (a fill takes no
multiple of its time with small tiles), and every table ends with its keys."""
import numpy as np
import pytest
import torch

from paper_1605_05236_gb300 import ck, inputs
from paper_1605_05236_gb300.multi import MULTI_TILE, MultiTable

pytestmark = pytest.mark.gpu


def test_large_tiles_over_small_tables():
    rng = np.random.default_rng(4)
    n = 2048
    bins, slots = rng.integers(100, 2500, n), rng.choice([4, 8], n)
    n_keys = (bins * slots * 0.9).astype(np.int64)
    keys, _ = inputs.distinct_keys(int(n_keys.sum()), 79)
    kt, vt = ck.as_u32_tensor(keys), ck.as_u32_tensor(inputs.values_for(keys))
    ms = {}
    for tile in (1000, 4096, 6000, 1 << 22):
        m = MultiTable(bins, slots, n_keys, ck.QUEUE, seed=9)
        m.set_param(MULTI_TILE, tile)
        st = torch.full((len(keys),), 99, dtype=torch.uint8, device="cuda")
        g = m.capture(kt, vt, st)
        times = []
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.launch()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        ms[tile] = min(times)
        assert bool((st == ck.ST_OK).all())
        assert m.stats()["size"] == len(keys)
        for i in (0, 1, n - 1):
            a = int(m.offsets[i])
            k = keys[a:a + n_keys[i]]
            assert m.contents(i) == dict(zip(k.tolist(), inputs.values_for(k).tolist()))
        g.close()
        m.close()
    assert max(ms.values()) < 4 * min(ms.values()), ms
