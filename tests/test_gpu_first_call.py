"""The first insertion a program makes pays for loading its kernel, but not for
unpacking compressed device code (10-11 ms a translation unit)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = """
import time, torch
from paper_1605_05236_gb300 import ck, inputs
keys, _ = inputs.distinct_keys(1000, 3)
kt, vt = ck.as_u32_tensor(keys), ck.as_u32_tensor(keys)
for B in (4, 8):
    t = ck.CuckooTable(1 << 12, B, 2, ck.QUEUE, seed=3)
    torch.cuda.synchronize()
    a = time.perf_counter()
    t.insert_batch(kt, vt)
    torch.cuda.synchronize()
    print((time.perf_counter() - a) * 1e3)
"""


def test_first_insert_call_does_not_unpack_code():
    best = [1e9, 1e9]
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        best = [min(x, float(y)) for x, y in zip(best, r.stdout.split())]
    assert max(best) < 6.0, best
