"""A stream call of a batched growth that fails on the host (by a preloaded
fake of it): the call returns GGA_ERR_CUDA with no growth kernel left running,
and the arrays can be cleared and grown again -- against the oracle."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "cuda", "fail_stream_call.c")
OUT = os.path.join(HERE, "cuda", "_build", "libfail_stream_call.so")

CHILD = """
import ctypes, sys
sys.path[:0] = [{root!r}, {here!r}]
import torch
import oracle
from paper_2209_00103_gb300 import gga
from paper_2209_00103_gb300 import workloads as wl
from harness import assert_same_state

fail_after = ctypes.CDLL({lib!r}).fail_after
thr = wl.poisson1_thresholds()
pool = gga.GGAPool(1 << 28, 256)
jobs, refs = [], []
for i, (E, target) in enumerate([(4, 300000), (8, 200000), (16, 90000), (4, 500)]):
    jobs.append((gga.GGArray(1, 256, 64, E, shared_pool=pool),
                 gga.make_gen_spec(i, "poisson", (1, 2, 3), thresholds=thr), target))
    o = oracle.OracleGGArray(1, 256, 64, E)
    o.grow_to_target(i, "poisson", (1, 2, 3), target, thresholds=thr)
    refs.append(o)
batch = gga.GGABatch(jobs)
batch.grow()
torch.cuda.synchronize()
calls = 0
for which in (0, 1):
    for n in range(1, 30):
        batch.clear()
        fail_after(which, n)
        rc = gga.load_library().gga_batch_grow(batch.h, None)
        fail_after(which, 0)
        if rc == gga.GGA_OK:      # it makes fewer than n such calls
            break
        assert rc == 5, rc
        calls += 1
        batch.clear()
        batch.grow()
        for (g, _, _), o in zip(jobs, refs):
            assert_same_state(g, o)
assert calls >= 6, calls
print("failed calls:", calls)
batch.close()
for g, _, _ in jobs:
    g.close()
pool.close()
"""


def test_a_failed_stream_call_leaves_a_usable_batch():
    os.makedirs(os.path.dirname(OUT), exist_ok=True)
    subprocess.run(["gcc", "-O2", "-shared", "-fPIC", "-o", OUT, SRC, "-ldl"], check=True)
    code = CHILD.format(root=os.path.dirname(HERE), here=HERE, lib=OUT)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=OUT))
    assert r.returncode == 0, r.stdout + r.stderr
    assert "failed calls:" in r.stdout
