"""Counts whose mean is well above one per thread and round: passes that leave
in several parts, clipped in the middle of one, cut short by the pool, for
every payload size and thread count, by the generated insertion and by the
batch -- against the oracle; and what they cost beside counts of mean one."""

import math

import numpy as np
import pytest
import torch

import oracle
from paper_2209_00103_gb300 import gga
from paper_2209_00103_gb300 import workloads as wl

from harness import assert_same_state

pytestmark = pytest.mark.gpu

COEFFS = ((1 << 40) | 0x10001, 0x9E3779B97F4A7, 7)


def poisson(mean):
    """16 thresholds of a Poisson distribution (cut off at 16)."""
    t, c, p = [], 0.0, math.exp(-mean)
    for k in range(16):
        c += p
        t.append(min((1 << 32) - 1, int(c * 2**32)))
        p *= mean / (k + 1)
    return np.array(t, dtype=np.uint32)


TABLES = {
    "3": poisson(3),
    "6": poisson(6),
    "always 16": np.zeros(16, dtype=np.uint32),
    "16 or none": np.full(16, 1 << 30, dtype=np.uint32),              # in bursts
    "unsorted": poisson(4)[::-1].copy(),
}


@pytest.mark.parametrize("E", [4, 8, 16])
@pytest.mark.parametrize("T", [1, 33, 100, 256, 257, 512, 700, 1024])
@pytest.mark.parametrize("table", TABLES)
def test_generated_insertion(E, T, table):
    thr = TABLES[table]
    for L, B, R in ((2, 64, 11), (1, 2, 9)):
        g = gga.GGArray(L, T, B, E, 2 * L * T * R * 16 * 2 * E + L * 64 * 256 + (1 << 20))
        o = oracle.OracleGGArray(L, T, B, E)
        for round0 in (0, R):
            g.insert_generated(gga.make_gen_spec(3, "poisson", COEFFS, round0=round0, thresholds=thr), R)
            o.insert_generated(3, "poisson", COEFFS, round0, R, thresholds=thr)
        assert_same_state(g, o)
        g.close()
        o.close()


@pytest.mark.parametrize("E", [4, 8, 16])
@pytest.mark.parametrize("T", [33, 256, 300, 600, 1000])
def test_batch(E, T):
    """Short chains and ones a cluster grows, clipped wherever the target falls."""
    arrays, jobs, refs = [], [], []
    for i, (table, rounds) in enumerate((t, r) for t in TABLES for r in (1, 7, 150)):
        thr = TABLES[table]
        mean = float(np.sum(1.0 - thr / 2.0**32))
        target = int(T * rounds * mean) - 3 * i
        g = gga.GGArray(1 + i % 2, T, (64, 4)[i % 2], E, 8 * max(target, 64) * E + (1 << 20))
        o = oracle.OracleGGArray(1 + i % 2, T, (64, 4)[i % 2], E)
        jobs.append((g, gga.make_gen_spec(i, "poisson", COEFFS, round0=i, thresholds=thr), target))
        o.grow_to_target(i, "poisson", COEFFS, target, round0=i, thresholds=thr)
        refs.append(o)
    batch = gga.GGABatch(jobs)
    batch.grow()
    for (g, _, _), o in zip(jobs, refs):
        assert_same_state(g, o)
    batch.close()
    for (g, _, _), o in zip(jobs, refs):
        g.close()
        o.close()


@pytest.mark.parametrize("T", [256, 512])
def test_a_full_pool_keeps_whole_rounds(T):
    B, E, R, thr = 64, 4, 40, TABLES["6"]
    cap = B * (2 ** 9 - 1)
    g = gga.GGArray(1, T, B, E, cap * E)
    g.insert_generated(gga.make_gen_spec(9, "poisson", COEFFS, thresholds=thr), R)
    n, rc = g.size()
    assert rc == gga.GGA_ERR_POOL_EXHAUSTED
    spec = wl.InsertSpec(L=1, T=T, E=E, seed=9, dist="poisson", rounds=R, coeffs=COEFFS, thresholds=thr)
    ends = np.cumsum(spec.counts().reshape(R, T).sum(axis=1))
    assert ends[-1] > cap and n == int(ends[ends <= cap].max())
    o = oracle.OracleGGArray(1, T, B, E)
    o.insert_generated(9, "poisson", COEFFS, 0, R, thresholds=thr)
    assert np.array_equal(g.flatten().cpu().numpy().view(np.uint32)[:n], o.flatten()[:n])
    g.close()
    o.close()


def microseconds(call):
    best = math.inf
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


@pytest.mark.parametrize("T,most", [(256, 2.0), (512, 2.6), (1024, 2.6)])
def test_three_elements_a_draw_cost_no_more_than_as_many_draws(T, most):
    """Time of 2^24 draws of mean 3 against mean 1; with the elements that do
    not fit a stage for mean one written one by one: 2.6, 4.3 and 3.7."""
    L, E = 1024, 4
    R = (1 << 24) // (L * T)
    g = gga.GGArray(L, T, 1024, E, 2 << 30)

    def grow(mean):
        g.clear()
        g.insert_generated(gga.make_gen_spec(7, "poisson", COEFFS, thresholds=poisson(mean)), R)

    assert microseconds(lambda: grow(3)) < most * microseconds(lambda: grow(1))
    assert g.last_error() == gga.GGA_OK
    g.close()


def test_blocks_of_256_threads_draw_for_themselves_alone():
    """A batch of 600 LFVectors by 256 threads each against 1024: as many draws
    (drawing for 1024 threads whatever T is took three times as long)."""
    def grow(T):
        pool = gga.GGAPool(1 << 30, 1024)
        arrays = [gga.GGArray(1, T, 8192, 4, shared_pool=pool) for _ in range(600)]
        batch = gga.GGABatch([(g, gga.make_gen_spec(a, "poisson", COEFFS, thresholds=poisson(1)), 100_000)
                              for a, g in enumerate(arrays)])

        def call():
            batch.clear()
            batch.grow()

        t = microseconds(call)
        batch.close()
        for g in arrays:
            assert g.size() == (100_000, gga.GGA_OK)
            g.close()
        pool.close()
        return t

    assert grow(256) < 2.3 * grow(1024)
