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


@pytest.mark.parametrize("newcap,atoms", [(256, 1 << 24), (512, 1 << 23), (1024, 1 << 22), (2048, 1 << 21)])
@pytest.mark.parametrize("ncode", [1, 27, 63, 125])
def test_sort_keys_of_the_cluster_builder(lib, newcap, atoms, ncode):
    """Keys of 32 bits: (atom, image) codes while they fit, then the atom alone
    up to 2^32 / newcap atoms, of which 2^24 at 9 moments; never refused below
    that (with 27 codes the builder used to end at 621,378 atoms)."""
    f = lib.cluster_key_codes
    f.argtypes = [ctypes.c_int] * 3
    f.restype = ctypes.c_int
    last = (atoms - 1) // ncode  # codes fit up to here
    assert f(last, ncode, newcap) == ncode and last * ncode * newcap < 2 ** 32
    if ncode > 1:
        assert f(last + 1, ncode, newcap) == 0
        assert f(atoms, ncode, newcap) == 0
        assert ((atoms - 1) * newcap + newcap - 1) < 2 ** 32
    assert f(atoms + 1, ncode, newcap) == -1
