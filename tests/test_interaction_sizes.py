"""Shared memory of an interaction block (host): calls that fit with a 32-bit code per column fit
although the columns are padded to packs of eight, or twice as many."""
import ctypes

import pytest

import paper_2511_09376_gb300 as wdf

SHARED = 232_448


@pytest.mark.parametrize("depth", range(2, 9))
def test_largest_ensembles_fit(depth):
    f = getattr(ctypes.CDLL(wdf.library_path()), "_ZN3wdf13iv_smem_bytesEiiiib")
    f.argtypes, f.restype = [ctypes.c_int] * 4 + [ctypes.c_bool], ctypes.c_size_t
    words = ((1 << depth) - 1 + 31) // 32
    for columns in (1, 2, 7, 8, 9, 40, 127, 300, 999, 5000):
        codes = -(-4 * columns // 16) * 16
        trees = (SHARED - codes) // (4 * words)
        assert codes + -(-4 * words * trees // 16) * 16 <= SHARED
        assert f(depth, columns, trees, -(-columns // 8) * 8, False) <= SHARED
        assert f(depth, columns, trees, 2 * columns, False) <= SHARED
