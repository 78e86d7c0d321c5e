"""Batched appends to arrays of any number of LFVectors: few (a warp takes the
buckets of each), many (a lane each), first appends and appends that need no
bucket, some LFVectors of a warp growing and others not, and a pool that runs
out -- against the oracle; and what many LFVectors cost."""

import numpy as np
import pytest

import oracle
from paper_2209_00103_gb300 import gga

from harness import assert_same_state
from test_gpu_count_means import microseconds

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [4, 16])
@pytest.mark.parametrize("L", [1, 7, 8, 9, 31, 33, 255, 256, 257, 1000, 2100])
def test_appends_equal_the_oracle(L, E):
    rng = np.random.default_rng(L)
    pool = gga.GGAPool(1 << 30, 256)
    Bs = (64, 4096, 512)
    arrays = [gga.GGArray(L, 32, B, E, shared_pool=pool) for B in Bs]
    refs = [oracle.OracleGGArray(L, 32, B, E) for B in Bs]
    try:
        # Shares that differ by one put some LFVectors past a bucket's end and others not.
        for step, per in enumerate([1, 63, 64, 1, 900, 0, 2500]):
            ns = [per * L + int(rng.integers(0, L + 1)) for _ in Bs]
            gga.gga_append_batch([(g, n, 10 * step + a) for a, (g, n) in enumerate(zip(arrays, ns))])
            for a, (o, n) in enumerate(zip(refs, ns)):
                o.append(n, 10 * step + a)
        for g, o in zip(arrays, refs):
            assert_same_state(g, o)
    finally:
        for g, o in zip(arrays, refs):
            g.close()
            o.close()
        pool.close()


@pytest.mark.parametrize("L", [3, 40, 600])
def test_a_full_pool_gives_whole_shares(L):
    B, E, per = 64, 4, 60
    pool = gga.GGAPool(L * B * E + (L // 2) * 2 * B * E, 256)   # second buckets for half of the LFVectors
    g = gga.GGArray(L, 32, B, E, shared_pool=pool)
    gga.gga_append_batch([(g, L * per, 1)])
    gga.gga_append_batch([(g, L * per, 2)])
    n, rc, sizes, _ = g.sizes_caps()
    assert rc == gga.GGA_ERR_POOL_EXHAUSTED
    sizes = sizes.cpu().numpy()
    assert set(sizes.tolist()) == {per, 2 * per} and int((sizes == 2 * per).sum()) == L // 2
    assert n == sizes.sum()
    flat = g.flatten().cpu().numpy().view(np.uint32)[:n]
    at = 0
    for l, s in enumerate(sizes):
        for tag in range(1, 1 + s // per):
            want = (tag << 24) + (l << 20) + np.arange(per)
            assert np.array_equal(flat[at:at + per], want.astype(np.uint32))
            at += per
    g.close()
    pool.close()


def test_many_lfvectors_cost_little():
    """Appends of one element per LFVector to 4 arrays of 4096 LFVectors, beside
    4 of 16 (with a warp for each LFVector: 45 times as long)."""
    def append(L):
        pool = gga.GGAPool(256 << 20, 1024)
        arrays = [gga.GGArray(L, 32, 1024, 4, shared_pool=pool) for _ in range(4)]
        reqs = [(g, L, a) for a, g in enumerate(arrays)]
        t = microseconds(lambda: [gga.gga_append_batch(reqs) for _ in range(4)])
        for g in arrays:
            assert g.size() == (36 * L, gga.GGA_OK)
            g.close()
        pool.close()
        return t

    assert append(4096) < 18 * append(16)
