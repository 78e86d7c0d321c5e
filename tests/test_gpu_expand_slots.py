"""gga_push_expand gives a thread one slot or several by the number of
LFVectors, and loads several as 128-bit words when T is a
multiple of them and both buffers are 16-byte aligned, element by element
otherwise, and each round's inputs ahead of the push that uses them: thread
counts around the slots, rounds around the rounds of a push, buffers off
their 16-byte boundary, counts past the two copies stored without a loop and
pushes larger than the stage, against the oracle's insertion of the same."""

import numpy as np
import pytest

import oracle
from paper_2209_00103_gb300 import gga

from harness import assert_same_state, counts_to_dev, packed_values, values_to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [4, 8, 16])
@pytest.mark.parametrize("T,R", [(1, 1), (2, 5), (3, 4), (4, 3), (30, 9), (128, 2), (132, 7), (509, 5), (512, 9)])
@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("L", [3, 200])               # one slot per thread up to one block per SM, then several
def test_slots_rounds_and_alignment(E, T, R, off, L):
    B = 8
    rng = np.random.default_rng(E * 1000 + T)
    counts = rng.integers(0, 3, size=(R, L, T)).astype(np.uint32)
    counts[0] = rng.integers(0, 9, size=(L, T))        # past two copies; a push past its stage for large T
    inputs = packed_values(R * L * T, E, seed=T)
    g = gga.GGArray(L, T, B, E, 16 * (int(counts.sum()) + B * L) * E + L * 64 * 256 + (1 << 20))
    o = oracle.OracleGGArray(L, T, B, E)
    x = values_to_dev(inputs, E, off)
    for _ in range(2):
        g.push_expand(counts_to_dev(counts, off), x.reshape((R, L, T) + tuple(x.shape[1:])))
        o.insert(counts, np.repeat(inputs, counts.reshape(-1)))
    assert_same_state(g, o)
    g.close()
    o.close()
