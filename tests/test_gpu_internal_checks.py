"""Parts of the library that its entry points reach only in passing: the
reciprocals that stand in for divisions, and the radix sort's tiles that count
the keys before them themselves instead of waiting for the tiles before."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2608_14266_gb300 import _lib
    assert torch.cuda.is_available()
    return _lib.lib()


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_reciprocals(lib, seed):
    """One rounding of the result (1 in these units) and what the last step leaves:
    2^-66 before the pivot's rounding, 2^-94 before the count's."""
    worst = (ctypes.c_double * 2)()
    assert lib.ba_check_reciprocals(0, 40_000_000, seed, worst) == 0
    assert 0.9 < worst[0] <= 1 + 2.0**-12
    assert 0.9 < worst[1] <= 1 + 2.0**-30


@pytest.mark.parametrize("n", [1, 2, 4096, 4097, 12289, 700_001, 3_000_000])
@pytest.mark.parametrize("bits", [0, 3, 16, 30, 36, 64])
@pytest.mark.parametrize("wait", [0, 1])
def test_sort(lib, n, bits, wait):
    """Without a wait, the tiles whose predecessors have not published count the
    keys themselves: full and ragged tiles, one digit to eight."""
    bad = ctypes.c_uint64()
    for seed in (1, 2):
        assert lib.ba_check_sort(0, n, bits, wait, seed, ctypes.byref(bad)) == 0
        assert bad.value == 0


def test_bad_arguments(lib):
    out = (ctypes.c_double * 2)()
    bad = ctypes.c_uint64()
    assert lib.ba_check_reciprocals(0, 0, 1, out) == 1
    assert lib.ba_check_reciprocals(0, 10, 1, None) == 1
    assert lib.ba_check_sort(0, 0, 8, 0, 1, ctypes.byref(bad)) == 1
    assert lib.ba_check_sort(0, 10, 65, 0, 1, ctypes.byref(bad)) == 1
    assert lib.ba_check_sort(0, 10, 8, 0, 1, None) == 1
