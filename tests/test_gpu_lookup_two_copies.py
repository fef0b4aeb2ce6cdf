"""A key stored twice in one bin: a lookup answers with the copy in the lowest
slot, wherever the copies lie in the bin and wherever the key stands in the
batch (8-slot bins are read by pairs of lanes, half a bin each)."""
import numpy as np
import pytest

from paper_1605_05236_gb300 import ck, inputs
from table_checks import bins_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,slots", [(8, (0, 4)), (8, (3, 7)), (8, (1, 2)), (8, (5, 6)), (4, (0, 3))])
@pytest.mark.parametrize("choice", [0, 1])
def test_lowest_slot_wins(B, slots, choice):
    bins = 64
    keys, _ = inputs.distinct_keys(400, 8)
    home = bins_np(keys, bins, 2)[:, choice].astype(np.int64)
    keys = keys[np.unique(home, return_index=True)[1]]  # one key a bin
    home = bins_np(keys, bins, 2)[:, choice].astype(np.int64)
    rec = np.full(bins * B, 0xFFFFFFFFFFFFFFFF, dtype=np.uint64)
    for i, s in enumerate(slots):
        rec[home * B + s] = (keys.astype(np.uint64) << np.uint64(32)) | np.uint64(100 + i)
    t = ck.CuckooTable(bins, B, 2, ck.QUEUE, seed=1)
    t.import_snapshot(rec, np.zeros(bins, dtype=np.uint32))
    probe = np.repeat(keys, 3)  # every key at even and odd places
    v, f = t.lookup(ck.as_u32_tensor(probe))
    assert bool((f == 1).all())
    assert (ck.u32_numpy(v) == 100).all()
