"""gga_push_generated plays four threads of an LFVector per thread and stages
each push in shared memory: thread counts around the four slots, one warp and
more than four warps, first buckets smaller than a 16-byte group, pushes
larger than the stage (geometric counts), and a pool that runs out, against
the oracle."""

import numpy as np
import pytest

import oracle
from paper_2209_00103_gb300 import gga
from paper_2209_00103_gb300 import workloads as wl

from harness import assert_same_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 3, 4, 5, 31, 127, 128, 129, 512, 513, 1023, 1024])
@pytest.mark.parametrize("dist,E,B", [("bernoulli", 4, 64), ("uniform3", 8, 1), ("geometric", 4, 2),
                                      ("poisson", 16, 16)])
def test_thread_counts_and_payloads(T, dist, E, B):
    thr = wl.poisson1_thresholds() if dist == "poisson" else None
    L, R, coeffs = 5, 9, (1 << 33 | 7, 1 << 20, 1 << 19)
    g = gga.GGArray(L, T, B, E, L * T * R * 8 * E + L * 64 * 256 + (1 << 20))
    o = oracle.OracleGGArray(L, T, B, E)
    for round0 in (0, R):
        g.push_generated(gga.make_gen_spec(11, dist, coeffs, round0=round0, thresholds=thr), R)
        o.insert_generated(11, dist, coeffs, round0, R, thresholds=thr)
        assert_same_state(g, o)
    g.close()
    o.close()


def test_a_pool_that_runs_out_keeps_whole_rounds():
    L, T, B, E, R = 1, 200, 64, 4, 40
    g = gga.GGArray(L, T, B, E, 7 * B * E + 256)          # three buckets of 64, 128, 256 elements
    g.push_generated(gga.make_gen_spec(5, "uniform3", (10, 1 << 20, 1)), R)
    o = oracle.OracleGGArray(L, T, B, E)
    fits = 0
    while True:
        p = oracle.OracleGGArray(L, T, B, E)
        p.insert_generated(5, "uniform3", (10, 1 << 20, 1), 0, fits + 1)
        if p.size() > 7 * B:
            p.close()
            break
        fits += 1
        p.close()
    o.insert_generated(5, "uniform3", (10, 1 << 20, 1), 0, fits)
    n, rc = g.size()
    assert rc == gga.GGA_ERR_POOL_EXHAUSTED and n == o.size()
    flat = g.flatten().cpu().numpy().view(np.uint32)[:n]
    assert np.array_equal(flat, o.flatten())
    g.close()
    o.close()
