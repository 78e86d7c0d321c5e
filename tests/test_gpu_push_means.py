"""Pushes of counts whose mean is well above one: the stage that holds them,
pushes larger than it, and counts no stage is made for -- gga_push_generated
against the oracle; and what they cost beside counts of mean one."""

import pytest

import oracle
from paper_2209_00103_gb300 import gga

from harness import assert_same_state
from test_gpu_count_means import COEFFS, TABLES, microseconds, poisson

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [4, 8, 16])
@pytest.mark.parametrize("T", [1, 33, 128, 129, 256, 500, 1024])
@pytest.mark.parametrize("table", TABLES)
def test_push_generated(E, T, table):
    thr = TABLES[table]
    for L, B, R in ((2, 64, 7), (1, 2, 5)):
        g = gga.GGArray(L, T, B, E, 2 * L * T * R * 16 * 2 * E + L * 64 * 256 + (1 << 20))
        o = oracle.OracleGGArray(L, T, B, E)
        for round0 in (0, R):
            g.push_generated(gga.make_gen_spec(3, "poisson", COEFFS, round0=round0, thresholds=thr), R)
            o.insert_generated(3, "poisson", COEFFS, round0, R, thresholds=thr)
        assert_same_state(g, o)
        g.close()
        o.close()


@pytest.mark.parametrize("T,most", [(256, 2.2), (512, 3.0), (1024, 2.8)])
def test_six_elements_a_draw_cost_no_more_than_as_many_draws(T, most):
    """Time of 2^24 draws of mean 6 against mean 1; with a stage for mean one:
    3.2, 4.8 and 4.5."""
    L, E = 1024, 4
    R = (1 << 24) // (L * T)
    g = gga.GGArray(L, T, 1024, E, 4 << 30)

    def grow(mean):
        g.clear()
        g.push_generated(gga.make_gen_spec(7, "poisson", COEFFS, thresholds=poisson(mean)), R)

    assert microseconds(lambda: grow(6)) < most * microseconds(lambda: grow(1))
    assert g.last_error() == gga.GGA_OK
    g.close()
