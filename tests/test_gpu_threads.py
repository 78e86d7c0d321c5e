"""Host threads that insert into arrays of their own at once, whose shapes
take the same kernel with different amounts of shared memory."""

import threading

import numpy as np
import pytest
import torch

import oracle
from paper_2209_00103_gb300 import gga

from harness import assert_same_state

pytestmark = pytest.mark.gpu

COEFFS = (1, 1 << 20, 1 << 19)


@pytest.mark.parametrize("push,E,shapes", [(False, 4, (256, 8, 129, 33)), (False, 16, (1024, 520, 800, 513)),
                                           (True, 16, (1024, 790, 900, 820))])
def test_inserts_from_several_threads(push, E, shapes):
    calls, failed = 400, []
    arrays = [gga.GGArray(3, T, 64, E, 256 << 20) for T in shapes]
    streams = [torch.cuda.Stream() for _ in shapes]
    torch.cuda.synchronize()
    start = threading.Barrier(len(shapes))

    def work(k):
        start.wait()
        try:
            for i in range(calls):
                spec = gga.make_gen_spec(7 + k, "uniform3", COEFFS, round0=i)
                (arrays[k].push_generated if push else arrays[k].insert_generated)(spec, 1, stream=streams[k])
        except gga.GGAError as e:
            failed.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(shapes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for k, T in enumerate(shapes):
        o = oracle.OracleGGArray(3, T, 64, E)
        o.insert_generated(7 + k, "uniform3", COEFFS, 0, calls)
        assert_same_state(arrays[k], o)
        o.close()
        arrays[k].close()
