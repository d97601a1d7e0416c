"""Index arithmetic of the kernels at the ends of its range, on the host (compiled with the library's own
headers): the bin of a pair for any alpha, and the offsets of single columns in a vector beyond 2^31 entries."""
import ctypes
import os

import pytest

from native_access import NVCC, compile_cuda

pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc is missing")

PAIRS = r"""
#include "mh_internal.cuh"
#include "pair64.cuh"
// smallest and largest bin over the first and last high words of every bin and of the cut; -1: table unused
extern "C" int bins(double alpha, int* lo, int* hi) {
    const mh_pair_tab T = mh_pair_tab_make(nullptr, alpha);
    *lo = 1 << 30;
    *hi = -(1 << 30);
    if (T.hi0 > T.hi_cut) return -1;
    for (long h = T.hi0; h <= T.hi_cut; h += 1 << (20 - PT_BITS_FAR)) {
        const int b = mh_pair_bin((int)h, T);
        *lo = *lo < b ? *lo : b;
        *hi = *hi > b ? *hi : b;
    }
    const int b = mh_pair_bin(T.hi_cut, T);
    *hi = *hi > b ? *hi : b;
    return PT_BINS;
}
"""

COLUMNS = r"""
#include "volume.cu"
extern "C" long column_offset(long at) {
    ColBuild b(1);
    b.open(0);
    b.add(1, {1.0}, at);
    b.close();
    return b.last > (long)UINT32_MAX ? -1 : (long)b.src[0];
}
"""


def test_pair_bins_stay_inside_the_table():
    lib = compile_cuda(PAIRS)
    lib.bins.argtypes = [ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p]
    used = 0
    for e in list(range(-320, 309, 4)) + [308.2]:
        alpha = 10.0 ** e
        lo, hi = ctypes.c_int(), ctypes.c_int()
        n = lib.bins(alpha, ctypes.byref(lo), ctypes.byref(hi))
        if n < 0:
            assert not 1e-140 < alpha < 1e140
            continue
        used += 1
        assert 0 <= lo.value and hi.value < n, (alpha, lo.value, hi.value)
    lo, hi = ctypes.c_int(), ctypes.c_int()
    assert lib.bins(float("inf"), ctypes.byref(lo), ctypes.byref(hi)) < 0
    assert used > 60


def test_column_offsets_beyond_two_to_the_31():
    lib = compile_cuda(COLUMNS)
    lib.column_offset.argtypes, lib.column_offset.restype = [ctypes.c_long], ctypes.c_long
    for at in (0, 2 ** 31 - 1, 2 ** 31, 3_000_000_000, 2 ** 32 - 1):
        assert lib.column_offset(at) == at
    assert lib.column_offset(2 ** 32) == -1
