"""The spawn kernel's block size follows the number of LFVectors (1024 threads
for few, 128 for many): every size of block, parents around a warp's 256 and
a pass, first buckets of one record, and a pool that runs out with blocks of
several groups of 1024 parents, against the oracle."""

import numpy as np
import pytest
import torch

import oracle
from paper_2209_00103_gb300 import gga
from paper_2209_00103_gb300 import workloads as wl

from harness import assert_same_state, counts_to_dev

pytestmark = pytest.mark.gpu


def pair(L, T, B, n0, pool_bytes):
    counts, recs = wl.split_counts(L, T, n0), wl.initial_records(n0)
    g, o = gga.GGArray(L, T, B, 16, pool_bytes), oracle.OracleGGArray(L, T, B, 16)
    g.insert(counts_to_dev(counts), torch.from_numpy(recs.view(np.int64).reshape(-1, 2)).cuda())
    o.insert(counts, recs.view(np.dtype((np.void, 16))))
    return g, o


@pytest.mark.parametrize("L,n0,generations", [(1, 255, 6), (1, 1025, 5), (2, 20000, 3), (160, 160 * 33, 4),
                                              (310, 310 * 300, 2), (620, 620 * 255, 2), (620, 620 * 1030, 1)])
@pytest.mark.parametrize("B", [1, 64])
@pytest.mark.parametrize("only_newborn", [False, True])
def test_every_block_size(L, n0, generations, B, only_newborn):
    g, o = pair(L, 32, B, n0, 64 * n0 * 16 * 4 + L * 64 * 256 + (64 << 20))
    born_d, born_o = torch.zeros(L, dtype=torch.int64, device="cuda"), np.zeros(L, dtype=np.uint64)
    for gen in range(generations):
        gga.gga_twophase_spawn(g.h, gen, 5, born_d if only_newborn else None)
        o.spawn(gen, 5, only_newborn, born_o)
        assert_same_state(g, o)
    g.close()
    o.close()


@pytest.mark.parametrize("L", [1, 200, 400, 700])
def test_a_pool_that_runs_out_keeps_groups_of_1024_parents(L):
    """Every LFVector has 6500 parents in buckets of 4096 and 8192 records, and
    the pool no more: about 6500 children each, of which those of the first
    groups of 1024 parents that fit in 3 * 4096 stay."""
    B, per = 4096, 6500
    g, o = pair(L, 512, B, per * L, (3 * B) * 16 * L)
    cap = 3 * B
    h = wl.splitmix_at(5, np.arange(per * L, dtype=np.uint64))          # generation 0: key = global index
    kids = wl.draw_counts("geometric", h).astype(np.int64).reshape(L, per)
    gga.gga_twophase_spawn(g.h, 0, 5)
    o.spawn(0, 5, False, np.zeros(L, dtype=np.uint64))
    n, rc, sizes, _ = g.sizes_caps()
    want = []
    for l in range(L):
        ends = [0] + [int(kids[l, :j].sum()) for j in range(1024, per, 1024)] + [int(kids[l].sum())]
        want.append(per + max(e for e in ends if per + e <= cap))
    assert sizes.cpu().tolist() == want
    assert (rc == gga.GGA_ERR_POOL_EXHAUSTED) == any(per + int(kids[l].sum()) > cap for l in range(L))
    offs, full = np.concatenate([[0], np.cumsum(want)]), o.offsets().astype(np.int64)
    flat, ref = g.flatten().cpu().numpy().reshape(-1, 2), o.flatten().view(np.int64).reshape(-1, 2)
    for l in range(0, L, max(1, L // 7)):
        assert np.array_equal(flat[offs[l]:offs[l + 1]], ref[full[l]:full[l] + want[l]])
    g.close()
    o.close()
