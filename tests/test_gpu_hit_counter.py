"""Queue-kicking's hit counter, which the device keeps as hits less occupied
slots: after deletes (fewer slots, the same hits), a snapshot taken and
restored in between, and serial insertions on top, the exported counters,
the slots and the duplicate marks equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_1605_05236_gb300 import ck, inputs
from test_gpu_parity import meta_fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bins,B,ghost,load", [(2, 4, False, 1.0), (1 << 9, 4, False, 0.95), (1 << 9, 4, True, 0.95),
                                               (777, 8, False, 0.97), (777, 8, True, 0.9)])
def test_hit_counter_through_deletes_and_a_snapshot(bins, B, ghost, load):
    n = inputs.load_target(bins * B, load)
    n_del = n // 3
    keys, _ = inputs.distinct_keys(n + n_del, 17)
    vals = inputs.values_for(keys)
    policy = ck.QUEUE | (ck.GHOST if ghost else 0)
    ref = oracle.OracleTable(bins, B, 2, policy, rng_seed=7, cap=500)
    t = ck.CuckooTable(bins, B, 2, policy, seed=7)

    def insert(table, a, b):
        ost = ref.insert(keys[a:b], vals[a:b])
        st = table.insert(ck.as_u32_tensor(keys[a:b]), ck.as_u32_tensor(vals[a:b]), serial=True)
        assert np.array_equal(st.cpu().numpy(), ost)

    insert(t, 0, n)
    gone = inputs.delete_keys(keys[:n], n_del, 3)
    assert np.array_equal(t.delete(ck.as_u32_tensor(gone)).cpu().numpy(), ref.delete(gone))
    slots, meta = t.export()
    u = ck.CuckooTable(bins, B, 2, policy, seed=7)
    u.import_snapshot(slots, meta)
    insert(u, n, n + n_del)
    slots, meta = u.export()
    e = ref.export()
    f = meta_fields(meta, B, 2)
    assert np.array_equal(slots, e["rec"])
    assert np.array_equal(f["hit"], e["hit"])
    assert np.array_equal(f["dup"], e["dup"])
    again = u.export()  # an export leaves the device's words as they were
    assert np.array_equal(again[0], slots) and np.array_equal(again[1], meta)
    torch.cuda.synchronize()
