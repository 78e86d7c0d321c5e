"""The device API with element types that a value is only explicitly converted
to (an enum class, a struct with an explicit constructor): it compiles without
a GPU, and the pushes equal the values; the value function is called for the
elements that are kept and no others; a count far past a bucket's end is
written bucket by bucket."""

import ctypes

import numpy as np
import pytest
import torch

from user_types_kernel import build_user, load_user


def test_explicit_element_types_compile():
    assert build_user()


@pytest.mark.gpu
@pytest.mark.parametrize("E", [4, 8])
@pytest.mark.parametrize("T,B", [(128, 64), (33, 1)])
def test_explicit_element_types(E, T, B):
    from paper_2209_00103_gb300 import gga
    L, R = 3, 4
    g = gga.GGArray(L, T, B, E, 8 << 20)
    lib = load_user()
    assert lib.user_push_typed(g.device_view(), L, T, R, E, None) == 0
    g.device_commit()
    n, rc = g.size()
    pushes = 2 * R + 3 * 2 + 1
    assert (n, rc) == (L * T * 3 * pushes, gga.GGA_OK)
    got = g.flatten().cpu().numpy().reshape(L, pushes, T * 3)
    one = (10 * np.arange(T)[:, None] + np.arange(3)[None, :]).reshape(-1)
    for l in range(L):
        assert (got[l] == l * 1000 + one).all()
    g.close()


@pytest.mark.gpu
@pytest.mark.parametrize("staged", [0, 1])
@pytest.mark.parametrize("T", [17, 128])
@pytest.mark.parametrize("case", ["all", "limit", "pool"])
def test_value_function_is_called_for_kept_elements(case, T, staged):
    from paper_2209_00103_gb300 import gga
    L, B = 1, 64
    g = gga.GGArray(L, T, B, 4, 64 * 7 * 4 if case == "pool" else 4 << 20)
    limit = 5 * T * 4 + 3 if case == "limit" else 1 << 40
    calls = torch.zeros(1, dtype=torch.int64, device="cuda")
    kept = torch.zeros(L, dtype=torch.int32, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert load_user().user_push_counted(g.device_view(), L, T, limit, staged, p(calls), p(kept), None) == 0
    g.device_commit()
    n, rc = g.size()
    assert rc == (gga.GGA_ERR_POOL_EXHAUSTED if case == "pool" and n < 5 * T * 9 else gga.GGA_OK)
    assert n == int(kept.sum()) == int(calls)
    if case == "limit":
        assert n == limit
    elif case == "all":
        assert n == 5 * T * 9
    g.close()


@pytest.mark.gpu
def test_one_large_count_costs_the_same_in_small_buckets():
    """2^20 elements of one thread into buckets from 64 elements on, beside one
    bucket that holds them all (a bucket search per element: 3 times as long)."""
    from paper_2209_00103_gb300 import gga
    from test_gpu_count_means import microseconds
    from user_kernel import load_user as load_push
    lib, n = load_push(), 1 << 20
    counts = torch.zeros(32, dtype=torch.int32, device="cuda")
    counts[5] = n

    def push(B):
        g = gga.GGArray(1, 32, B, 8, 64 << 20)

        def call():
            g.clear()
            assert lib.user_push_formula(ctypes.c_void_p(g.device_view()), ctypes.c_void_p(counts.data_ptr()), 1, 1,
                                         32, 1, None) == 0
            g.device_commit()

        t = microseconds(call)
        assert g.size() == (n, gga.GGA_OK)
        g.close()
        return t

    assert push(64) < 1.5 * push(n)
