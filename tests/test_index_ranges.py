"""Index arithmetic of the kernels at the ends of its range, on the host (compiled with the library's own
headers): the bin of a pair for any alpha."""
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
