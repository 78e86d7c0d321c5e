"""The prefix sums that end every insertion (offsets, 16 KB chunks) and the
pool's queue heads: numbers of LFVectors around one sweep of the finalize
step (up to four LFVectors per thread of its block) and sizes around bucket
and chunk edges, against the oracle; flatten and rw_b walk the chunk list."""

import numpy as np
import pytest

from paper_2209_00103_gb300 import gga

from harness import assert_same_state, insert_both, make_pair, packed_values

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [1, 31, 255, 257, 1024, 1025, 4097])
@pytest.mark.parametrize("B,E", [(1, 16), (256, 4), (4096, 8)])
def test_sizes_around_bucket_and_chunk_edges(L, B, E):
    edges = [0, 1, B, 3 * B, 7 * B, 16384 // E, 2 * 16384 // E]
    sizes = sorted({max(0, e + d) for e in edges for d in (-1, 0, 1)} | {0})
    if L > 300:
        sizes = [s for s in sizes if s <= 2 * B + 2] or sizes
    counts = np.resize(np.array(sizes, dtype=np.uint32), L).reshape(1, L, 1)
    n = int(counts.sum())
    g, o = make_pair(L, 1, B, E, pool_bytes=L * 64 * max(256, B * E) + (64 << 20))
    for rep in range(2):            # the second time buckets come from the pool's queues
        insert_both(g, o, counts, packed_values(n, E, seed=rep), E)
        assert_same_state(g, o)
        if E != 16:
            g.sweep(gga.GGA_RW_B, 3, 1)
            o.sweep_add(3, 1)
            assert_same_state(g, o)
        if rep == 0:
            held = g.memory()["pool_bump_bytes"]
            g.clear()
            assert g.size() == (0, gga.GGA_OK)
            o.close()
            _, o = make_pair(L, 1, B, E, pool_bytes=1 << 20)
    assert g.memory()["pool_bump_bytes"] == held
    g.close()
    o.close()


@pytest.mark.parametrize("T,R", [(16, 1), (16, 33), (16, 2045), (16, 2047), (16, 2049), (128, 130)])
def test_count_tiles_around_the_scan_by_the_last_block(T, R):
    """32 rows a tile (128 for T = 128): one tile, and 1023 to 1025 around the line."""
    L = 16
    for rounds in (R, R + 1):
        counts = (np.arange(rounds * L * T, dtype=np.uint64) * 2654435761 % 3).astype(np.uint32).reshape(rounds, L, T)
        n = int(counts.sum())
        g, o = make_pair(L, T, 64, 4, expected_elems=n)
        for _ in range(2):
            insert_both(g, o, counts, packed_values(n, 4), 4)
        assert_same_state(g, o)
        g.close()
        o.close()
