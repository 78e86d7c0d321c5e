"""Batched growth by clusters of blocks and by marks: LFVectors long enough
for a cluster's passes beside short ones, every payload size and count
distribution, thread counts below and at a block's virtual threads, first
buckets smaller than a lane's group, targets around the end of a pass, a
target reached in an earlier growth, and a pool that runs out in the middle
of a cluster's pass -- against the oracle."""

import numpy as np
import pytest
import torch

import oracle
from paper_2209_00103_gb300 import gga
from paper_2209_00103_gb300 import workloads as wl

from harness import assert_same_state

pytestmark = pytest.mark.gpu

DISTS = ["bernoulli", "uniform3", "geometric", "poisson"]
COEFFS = ((1 << 40) | 0x10001, 0x9E3779B97F4A7, 7)


@pytest.mark.parametrize("E", [4, 8, 16])
@pytest.mark.parametrize("T,B", [(1024, 256), (1000, 1), (64, 4), (33, 2)])
def test_long_and_short_chains(E, T, B):
    thr = wl.poisson1_thresholds()
    pool = gga.GGAPool(1 << 30, 256)
    jobs, refs = [], []
    # 64 rounds a block's pass of 8 make a chain of 8; clusters take 16 passes and more.
    targets = [T * 400 + 1, T * 200, T * 16, T * 8 + 1, T, 1, 0]
    for i, dist in enumerate(DISTS):
        for j, target in enumerate(targets):
            seed = 100 * i + j
            L = 2 if j == 1 else 1
            g = gga.GGArray(L, T, max(B, 256 // E), E, shared_pool=pool) if j % 2 else gga.GGArray(
                L, T, B, E, 64 * (target + 256) * E + (1 << 20))
            o = oracle.OracleGGArray(L, T, max(B, 256 // E) if j % 2 else B, E)
            t = thr if dist == "poisson" else None
            o.grow_to_target(seed, dist, COEFFS, target, round0=j, thresholds=t)
            jobs.append((g, gga.make_gen_spec(seed, dist, COEFFS, round0=j, thresholds=t), target))
            refs.append(o)
    batch = gga.GGABatch(jobs)
    try:
        batch.grow()
        for (g, _, _), o in zip(jobs, refs):
            assert_same_state(g, o)
        batch.grow()                     # every target is reached: nothing changes
        for (g, _, target), o in zip(jobs, refs):
            assert g.size() == (target, gga.GGA_OK)
        batch.clear()
        batch.grow()
        for (g, _, _), o in zip(jobs, refs):
            assert_same_state(g, o)
        s = torch.cuda.Stream()
        batch.capture(s)
        batch.replay(s)
        s.synchronize()
        for (g, _, _), o in zip(jobs, refs):
            assert_same_state(g, o)
    finally:
        # Also when a comparison fails: arrays before the pool they live in.
        batch.close()
        for (g, _, _), o in zip(jobs, refs):
            g.close()
            o.close()
        pool.close()


@pytest.mark.parametrize("dist", DISTS)
def test_a_pool_that_runs_out_in_a_cluster_keeps_whole_rounds(dist):
    T, B, E, seed = 512, 64, 4, 9
    thr = wl.poisson1_thresholds() if dist == "poisson" else None
    buckets = 11                                    # 64 * 2047 = 131,008 elements fit
    cap = B * (2 ** buckets - 1)
    g = gga.GGArray(1, T, B, E, cap * E)
    batch = gga.GGABatch([(g, gga.make_gen_spec(seed, dist, COEFFS, thresholds=thr), 4 * cap)])
    batch.grow()
    n, rc = g.size()
    assert rc == gga.GGA_ERR_POOL_EXHAUSTED
    o = oracle.OracleGGArray(1, T, B, E)
    o.grow_to_target(seed, dist, COEFFS, 2 * cap, thresholds=thr)
    # The most whole rounds that fit, from the counts themselves.
    spec = wl.InsertSpec(L=1, T=T, E=E, seed=seed, dist=dist, rounds=1200, coeffs=COEFFS, thresholds=thr)
    ends = np.cumsum(spec.counts().reshape(1200, T).sum(axis=1))
    assert ends[-1] > cap
    assert n == int(ends[ends <= cap].max())
    flat = g.flatten().cpu().numpy().view(np.uint32)[:n]
    assert np.array_equal(flat, o.flatten()[:n])
    batch.close()
    g.close()
    o.close()


@pytest.mark.parametrize("E", [4, 8, 16])
@pytest.mark.parametrize("dist", ["geometric", "poisson", "uniform3"])
@pytest.mark.parametrize("T", [1, 33, 256, 257, 512, 700, 1024])
def test_generated_insertion_of_every_shape(E, dist, T):
    thr = None
    if dist == "poisson":            # several thresholds inside one interval of the count table, one on its edge
        thr = np.array([1 << 23, 5 << 28, (5 << 28) + 1, (5 << 28) + 7, 0xFFFFFFF0, 0xFFFFFFFF], dtype=np.uint32)
    for L, B, R in ((3, 1, 19), (2, 64, 8)):
        g = gga.GGArray(L, T, B, E, 64 * L * T * R * E + L * 64 * 256 + (1 << 20))
        o = oracle.OracleGGArray(L, T, B, E)
        for round0 in (0, R):
            g.insert_generated(gga.make_gen_spec(3, dist, COEFFS, round0=round0, thresholds=thr), R)
            o.insert_generated(3, dist, COEFFS, round0, R, thresholds=thr)
        assert_same_state(g, o)
        g.close()
        o.close()
