"""Lookups of every table shape at sizes around a warp (8-slot bins are read by
pairs of lanes), with reserved keys beside present and absent ones, repeated
keys, and either output missing; a key stored twice is answered from its first
bin."""
import numpy as np
import pytest
import torch

from paper_1605_05236_gb300 import ck, inputs

pytestmark = pytest.mark.gpu

SHAPES = [(1 << 9, 4, 2, ck.QUEUE), (333, 8, 2, ck.QUEUE), (1 << 9, 8, 2, ck.RANDOM | ck.GHOST),
          (4001, 1, 3, ck.RANDOM), (1 << 12, 1, 4, ck.RATTLE)]


@pytest.mark.parametrize("bins,B,d,policy", SHAPES)
@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 63, 255, 256, 257, 1001])
def test_lookup_sizes(bins, B, d, policy, n):
    t = ck.CuckooTable(bins, B, d, policy, seed=5)
    keys, _ = inputs.distinct_keys(inputs.load_target(bins * B, 0.8) + 600, 12)
    have, absent = keys[:-600], keys[-600:]
    t.insert(ck.as_u32_tensor(have), ck.as_u32_tensor(inputs.values_for(have)))
    rng = np.random.default_rng(n)
    probe = np.where(rng.random(n) < 0.5, rng.choice(have, n), rng.choice(absent, n)).astype(np.uint32)
    probe[rng.random(n) < 0.15] = 0xFFFFFFFF
    want = np.isin(probe, have)
    v, f = t.lookup(ck.as_u32_tensor(probe))
    assert np.array_equal(f.cpu().numpy(), want.astype(np.uint8))
    assert np.array_equal(ck.u32_numpy(v), np.where(want, inputs.values_for(probe), 0).astype(np.uint32))
    L, kt = ck.load(), ck.as_u32_tensor(probe)
    only_v, only_f = torch.zeros_like(v), torch.zeros_like(f)
    assert L.ck_lookup_batch(t._h, ck._ptr(kt), n, ck._ptr(only_v), None, ck._stream(None)) == ck.OK
    assert L.ck_lookup_batch(t._h, ck._ptr(kt), n, None, ck._ptr(only_f), ck._stream(None)) == ck.OK
    assert torch.equal(only_v, v) and torch.equal(only_f, f)
    s = t.stats()
    assert s["lookups"] == 3 * n and s["lookup_hits"] == 3 * int(want.sum())


@pytest.mark.parametrize("B", [4, 8])
def test_first_bins_copy_wins(B):
    t = ck.CuckooTable(64, B, 2, ck.QUEUE, seed=1)
    keys, _ = inputs.distinct_keys(40, 2)
    kt = ck.as_u32_tensor(keys)
    for value in (1, 2):  # the second insertion of a key stores a second copy
        t.insert(kt, torch.full_like(kt, value), serial=True)
    slots, _ = t.export()
    v, f = t.lookup(kt)
    assert f.all()
    where = {}
    for i, r in enumerate(slots):
        if r != np.uint64(0xFFFFFFFFFFFFFFFF):
            where.setdefault(int(r >> np.uint64(32)), []).append((i // B, int(r & np.uint64(0xFFFFFFFF))))

    def mix(h):
        h ^= h >> 16
        h = h * 0x85EBCA6B & 0xFFFFFFFF
        h ^= h >> 13
        h = h * 0xC2B2AE35 & 0xFFFFFFFF
        return h ^ h >> 16

    for k, got in zip(keys.tolist(), v.tolist()):
        copies = where[k]
        assert len(copies) == 2
        first = [x for b, x in copies if b == mix(k ^ 0x9E3779B9) % 64]
        assert got == (first or [x for _, x in copies])[0]
