"""gga_push_expand with counts of neighbouring slots whose sum passes 32 bits:
the slots' thread pushes nothing in that round and the error is latched; all
other elements are there."""

import numpy as np
import pytest

import oracle
from paper_2209_00103_gb300 import gga

from harness import counts_to_dev, packed_values, values_to_dev

pytestmark = pytest.mark.gpu

HUGE = [(1 << 31, 1 << 31, 5, 0), ((1 << 32) - 1, 1, 0, 0), (1 << 30, 1 << 30, 1 << 30, 1 << 30), (7, 0, (1 << 32) - 4, 3)]


@pytest.mark.parametrize("E", [4, 8, 16])
@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("huge", HUGE)
def test_sums_past_32_bits(E, off, huge):
    L, T, R, B = 400, 64, 6, 64
    if E == 16:                                        # two slots a thread
        huge = next(p for p in (huge[:2], huge[2:]) if sum(p) >> 32) if any(
            sum(p) >> 32 for p in (huge[:2], huge[2:])) else ((1 << 32) - 1, 1)
    rng = np.random.default_rng(E)
    counts = rng.integers(0, 3, size=(R, L, T)).astype(np.uint32)
    want = counts.copy()
    for r, l, t in ((0, 0, 0), (3, 7, 60), (5, 399, 20)):
        t -= t % len(huge)
        counts[r, l, t:t + len(huge)] = huge
        want[r, l, t:t + len(huge)] = 0
    inputs = packed_values(R * L * T, E, seed=1)
    g = gga.GGArray(L, T, B, E, 16 * (int(want.sum()) + B * L) * E + L * 64 * 256 + (1 << 20))
    o = oracle.OracleGGArray(L, T, B, E)
    x = values_to_dev(inputs, E, off)
    g.push_expand(counts_to_dev(counts, off), x.reshape((R, L, T) + tuple(x.shape[1:])))
    o.insert(want, np.repeat(inputs, want.reshape(-1)))
    n, rc, sizes, _ = g.sizes_caps()
    assert rc == gga.GGA_ERR_INVALID and n == o.size()
    assert np.array_equal(sizes.cpu().numpy().astype(np.uint64), o.sizes())
    flat = g.flatten().cpu().contiguous().numpy().view(np.uint8).reshape(-1)[: n * E]
    assert flat.tobytes() == o.flatten().tobytes()
    g.close()
    o.close()
