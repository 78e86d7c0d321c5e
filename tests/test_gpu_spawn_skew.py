"""Spawning where some LFVectors hold far more records than the others: those
go to blocks of 1024 threads after the small blocks' kernel -- one or many of
them, next to each other, around the size that makes the difference, parents
of the last generation only, in a captured stream, in a pool that runs out --
against the oracle; and what skew costs."""

import numpy as np
import pytest
import torch

import oracle
from paper_2209_00103_gb300 import gga
from paper_2209_00103_gb300 import workloads as wl

from harness import assert_same_state, counts_to_dev
from test_gpu_count_means import microseconds

pytestmark = pytest.mark.gpu


def pair(sizes, pool_bytes, T=32, B=64, ref=True):
    L, n = len(sizes), int(np.sum(sizes))
    counts = np.zeros((1, L, T), dtype=np.uint32)
    counts[0] = (np.asarray(sizes) // T)[:, None] + (np.arange(T)[None, :] < (np.asarray(sizes) % T)[:, None])
    recs = wl.initial_records(n)
    g, o = gga.GGArray(L, T, B, 16, pool_bytes), None
    g.insert(counts_to_dev(counts), torch.from_numpy(recs.view(np.int64).reshape(-1, 2)).cuda())
    if ref:
        o = oracle.OracleGGArray(L, T, B, 16)
        o.insert(counts, recs.view(np.dtype((np.void, 16))))
    return g, o


def skewed(L, kind):
    sizes = np.full(L, 20)
    if kind == "one":
        sizes[L // 2] = 40000
    elif kind == "edges":                          # around 16384 records
        sizes[[0, 3, 5, L - 1]] = (16384, 16385, 16383, 20000)
    elif kind == "neighbours":                     # more than one for a block of the second kernel
        sizes[10:20] = 17000
        sizes[[0, 160, 320][: 1 + L // 320]] = 18000
        sizes[[152, 304]] = 16500
    elif kind == "none large":
        sizes[:] = 30
        sizes[7] = 0
    return sizes


@pytest.mark.parametrize("only_newborn", [False, True])
@pytest.mark.parametrize("L", [320, 650])
@pytest.mark.parametrize("kind", ["one", "edges", "neighbours", "none large"])
def test_spawn(L, kind, only_newborn):
    sizes = skewed(L, kind)
    g, o = pair(sizes, 64 * int(sizes.sum()) * 16 * 2 + L * 64 * 256 + (64 << 20))
    born_d, born_o = torch.zeros(L, dtype=torch.int64, device="cuda"), np.zeros(L, dtype=np.uint64)
    for gen in range(2):
        gga.gga_twophase_spawn(g.h, gen, 5, born_d if only_newborn else None)
        o.spawn(gen, 5, only_newborn, born_o)
        assert_same_state(g, o)
    if only_newborn:
        assert np.array_equal(born_d.cpu().numpy().astype(np.uint64), born_o)
    g.close()
    o.close()


def test_capture_and_replay():
    sizes = skewed(400, "neighbours")
    g, o = pair(sizes, 1 << 30)
    graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=s):
        gga.gga_twophase_spawn(g.h, 3, 5, stream=s)
    for _ in range(2):
        graph.replay()
        o.spawn(3, 5, False, np.zeros(400, dtype=np.uint64))
    torch.cuda.synchronize()
    assert_same_state(g, o)
    g.close()
    o.close()


def test_a_pool_that_runs_out_in_a_large_lfvector_keeps_groups_of_1024_parents():
    L, B, T = 400, 64, 32
    sizes = np.full(L, 20)
    sizes[9] = 30000
    per_small, cap = 2, 64 * 1023                  # the large one's buckets 0 .. 9 and two for each small one
    pool = cap * 16 + (L - 1) * 64 * (2 ** per_small - 1) * 16
    g, _ = pair(sizes, pool, T, B, ref=False)
    offs = np.concatenate([[0], np.cumsum(sizes)])
    kids = wl.draw_counts("geometric", wl.splitmix_at(5, np.arange(sizes.sum(), dtype=np.uint64))).astype(np.int64)
    # A second generation does not fit the large one: gen 0 takes it to about 60,000 of 65,472.
    gga.gga_twophase_spawn(g.h, 0, 5)
    n, rc, s1, _ = g.sizes_caps()
    assert rc == gga.GGA_OK
    s1 = s1.cpu().numpy()
    assert all(s1[l] == sizes[l] + kids[offs[l]:offs[l + 1]].sum() for l in range(L))
    offs1 = np.concatenate([[0], np.cumsum(s1)])
    keys = (np.uint64(1) << np.uint64(48)) | np.arange(offs1[9], offs1[10]).astype(np.uint64)
    kids1 = wl.draw_counts("geometric", wl.splitmix_at(5, keys)).astype(np.int64)
    gga.gga_twophase_spawn(g.h, 1, 5)
    n, rc, s2, _ = g.sizes_caps()
    assert rc == gga.GGA_ERR_POOL_EXHAUSTED
    ends = [0] + [int(kids1[:j].sum()) for j in range(1024, len(kids1), 1024)]
    assert int(s2[9]) == int(s1[9]) + max(e for e in ends if s1[9] + e <= cap)
    g.close()


def test_skew_costs_its_chain_and_no_more():
    """Half of the records in one LFVector, three generations: 1024 LFVectors beside
    120, which are all taken by blocks of 1024 threads (by a block of 128: 3
    times as long)."""
    def spawn(L):
        sizes = np.full(L, (1 << 18) // (L - 1))
        sizes[L // 2] = 1 << 18
        g, _ = pair(sizes, 4 << 30, 512, 1024, ref=False)
        start = g.flatten()[: int(sizes.sum())].clone()
        T = 512
        counts = np.zeros((1, L, T), dtype=np.uint32)
        counts[0] = (sizes // T)[:, None] + (np.arange(T)[None, :] < (sizes % T)[:, None])
        counts = counts_to_dev(counts)

        def call():
            g.clear()
            g.insert(counts, start)
            for gen in range(3):
                gga.gga_twophase_spawn(g.h, gen, 5)

        t = microseconds(call)
        assert g.last_error() == gga.GGA_OK
        g.close()
        return t

    assert spawn(1024) < 1.8 * spawn(120)
