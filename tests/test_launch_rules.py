"""CPU checks of rules that choose a launch (host code of libbopgb.so)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_1803_07491_gb300 import build
    return ctypes.CDLL(build.build())


@pytest.mark.parametrize("slots", [0, 1, 151, 152, 608, 100000])
@pytest.mark.parametrize("n_items", [1, 152, 609, 4000])
def test_no_more_ctas_than_scratch_slots(lib, slots, n_items):
    """A sweep whose Psi lies in global memory has one scratch slot per CTA,
    with a Psi store as without one: the grid is bounded in both cases."""
    f = lib.launch_max_ctas
    f.argtypes = [ctypes.c_int, ctypes.c_size_t, ctypes.c_size_t, ctypes.c_int]
    f.restype = ctypes.c_int
    slot = 217 * 208
    for extra in (0, 1, slot - 1):  # bytes beyond the last whole slot
        m = f(1, slots * slot + extra, slot, n_items)
        assert m == min(slots, n_items) and m * slot <= slots * slot + extra
    assert f(0, 0, slot, n_items) == n_items
