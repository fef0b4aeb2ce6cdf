"""No claim outlives its transaction: after workers have contended for tables
of two bins that are full or nearly so, with claim flags and with system-
transaction kick-outs whose moves fail now and then, one worker can fill every
slot.  (An insertion passes over a claimed slot, so a claim left behind keeps
its slot empty; in two bins any key may go to any slot.)"""
import numpy as np
import pytest
import torch

from paper_1605_05236_gb300 import inputs, txn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [txn.LOCAL_RETRY | txn.CLAIM, txn.LOCAL_RETRY | txn.CLAIM | txn.SYSTEM,
                                   txn.LOCAL_RETRY | txn.CLAIM | txn.SYSTEM | txn.QUEUE])
@pytest.mark.parametrize("B,W", [(8, 20), (4, 9)])
def test_every_slot_can_be_filled_afterwards(B, W, flags):
    bins, T, trials = 2, 60, 1024
    keys, _ = inputs.distinct_keys(W + bins * B, 23)
    tab = txn.TxnTable(bins, B, trials, seed=11)

    def run(op, key, workers, txns):
        dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
               for a in (op.astype(np.uint8), key.view(np.int32), inputs.values_for(key).view(np.int32))]
        out = tab.run(*dev, workers, txns, 1, flags)
        torch.cuda.synchronize()
        return out["status"].cpu().numpy()

    # each worker inserts its key and deletes it again, in turn
    run(np.tile([txn.TX_INSERT, txn.TX_DELETE], W * T // 2), np.repeat(keys[:W], T), W, T)
    s = tab.stats()
    run(np.full(W, txn.TX_DELETE), keys[:W], 1, W)  # what a given-up deletion left
    st = run(np.full(bins * B, txn.TX_INSERT), keys[W:], 1, bins * B)
    assert (st == 0).all(), (int((st != 0).sum()), s)
    for r in range(0, trials, 37):
        slots = tab.export(r)
        assert np.array_equal(np.sort((slots >> np.uint64(32)).astype(np.uint32)), np.sort(keys[W:]))
    tab.close()
