"""Pairs of transactions that read the bins each other writes, started
together: each inserts 48 keys and reads 48 absent keys, one in every bin the
other inserts into.  Neither changes what the other read, so with local
retries both commit at their first attempt, however long they have kept in
step."""
import numpy as np
import pytest
import torch

from paper_1605_05236_gb300 import inputs, txn
from table_checks import SEEDS, fmix32_np
import oracle

pytestmark = pytest.mark.gpu


def _bins(keys, bins, seed):  # trial 0's bins (power-of-two table)
    salt = oracle.splitmix64_at(seed) & 0xFFFFFFFF
    b0, b1 = (fmix32_np(keys ^ np.uint32(SEEDS[i] ^ salt)) % np.uint32(bins) for i in (0, 1))
    return b0, np.where(b1 == b0, (b1 + 1) % np.uint32(bins), b1)


@pytest.mark.parametrize("flags", [txn.LOCAL_RETRY, txn.LOCAL_RETRY | txn.CLAIM,
                                   txn.LOCAL_RETRY | txn.CLAIM | txn.SYSTEM])
@pytest.mark.parametrize("ins", [3, 12, 48])
def test_pairs_in_step_commit_at_once(flags, ins):
    bins, B, pairs, seed = 1 << 16, 8, 32, 5
    W, L = 2 * pairs, 2 * ins
    keys, _ = inputs.distinct_keys(1 << 20, 19)
    b0, b1 = _bins(keys, bins, seed)
    uniq = np.unique(b0, return_index=True)[1][:W * ins]  # inserted keys: distinct first bins, which are empty
    mine = uniq.reshape(W, ins)
    free = np.ones(len(keys), dtype=bool)
    free[uniq] = False
    cand = np.nonzero(free)[0]
    order = cand[np.argsort(b1[cand], kind="stable")]
    first = np.searchsorted(b1[order], np.arange(bins))
    first = order[np.minimum(first, len(order) - 1)]       # a key with second bin b, for every bin b that has one
    reads = first[b0[mine]]                                # ... for every bin written
    assert (b1[reads] == b0[mine]).all()
    other = reads.reshape(pairs, 2, ins)[:, ::-1].reshape(W, ins)
    key = np.concatenate([keys[mine], keys[other]], axis=1).reshape(-1)
    op = np.concatenate([np.full((W, ins), txn.TX_INSERT, np.uint8), np.full((W, ins), txn.TX_READ, np.uint8)],
                        axis=1).reshape(-1)
    tab = txn.TxnTable(bins, B, 1, seed=seed)
    dev = [torch.from_numpy(a).cuda() for a in (op, key.view(np.int32), inputs.values_for(key).view(np.int32))]
    for _ in range(4):
        tab.reset()
        out = tab.run(*dev, W, 1, L, flags)
        s = tab.stats()
        assert s["failed"] == 0 and s["commits"] == W, str(s)
        assert s["attempts"] == W, str(s)
        assert bool((out["status"] == 0).all())
        slots = tab.export(0)
        stored = np.sort((slots[slots != np.uint64(0xFFFFFFFFFFFFFFFF)] >> np.uint64(32)).astype(np.uint32))
        assert np.array_equal(stored, np.sort(keys[mine].reshape(-1)))
    tab.close()
