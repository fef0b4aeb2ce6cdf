"""Registers and spills of the kernels that fill tables, as the compiler prints
them for sm_103a: the queue-kicking fill of 4-slot tables (k_insert_walk, and
k_multi_walk in the batched form) without spills inside its register bound,
the searches whose first groups are in shared memory without spills, and the
search upserts (k_insert, 64 registers) without the several hundred bytes that
a loop of steps around a search costs them.  Cross-compiles, no GPU."""
import os
import re
import shutil
import subprocess
import tempfile
from concurrent.futures import ThreadPoolExecutor

import pytest

from paper_1605_05236_gb300 import build as ckbuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# source, mangled kernel and template arguments, registers and spill bytes at most
QUEUE, SORTED, BFS, HYBRID = 3, 2, 1, 5
BOUNDS = [
    ("ck_insert_b4.cu", "13k_insert_walkILi4ELi%dELb0E" % QUEUE, 80, 0),
    ("ck_insert_b4.cu", "13k_insert_walkILi4ELi%dELb0E" % SORTED, 128, 0),
    ("ck_insert_b8.cu", "13k_insert_walkILi8ELi%dELb0E" % SORTED, 128, 0),
    ("ck_multi.cu", "12k_multi_walkILi4ELi%dE" % QUEUE, 128, 0),
    ("ck_multi.cu", "12k_multi_walkILi8ELi%dE" % QUEUE, 128, 0),
] + [("ck_insert_b4.cu", "8k_insertILi4ELi%dELb0ELb0E" % p, 64, 200) for p in (BFS, SORTED, HYBRID)] \
  + [("ck_insert_b8.cu", "8k_insertILi8ELi%dELb0ELb0E" % p, 64, 400) for p in (BFS, SORTED, HYBRID)]


def _compile(src):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    with tempfile.TemporaryDirectory() as d:
        r = subprocess.run([nvcc] + ckbuild.ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xptxas", "-v",
                                                    "-I" + os.path.join(ROOT, "include"), "-I" + ckbuild.CSRC, "-c",
                                                    os.path.join(ckbuild.CSRC, src), "-o", os.path.join(d, "x.o")],
                           capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return (r.stdout + r.stderr).splitlines()


@pytest.mark.timeout(600)
def test_registers_and_spills():
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("nvcc not found")
    srcs = sorted({b[0] for b in BOUNDS})
    with ThreadPoolExecutor(len(srcs)) as ex:
        logs = dict(zip(srcs, ex.map(_compile, srcs)))
    bad = []
    for src, kernel, max_regs, max_spill in BOUNDS:
        lines = logs[src]
        at = next(i for i, l in enumerate(lines) if "Compiling entry function '" in l and kernel in l)
        tail = "\n".join(lines[at + 1:at + 5])
        stores = int(re.search(r"(\d+) bytes spill stores", tail).group(1))
        regs = int(re.search(r"Used (\d+) registers", tail).group(1))
        if regs > max_regs or stores > max_spill:
            bad.append((kernel, regs, stores))
    assert not bad, bad
