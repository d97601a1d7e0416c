"""A device buffer after a failed allocation (csrc/mh_internal.cuh): it holds nothing, so a later reserve
tries again instead of reporting room that is not there.  Host calls only: the request is larger than any
device, so the driver refuses it."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "mh_internal.cuh"
extern "C" void failed_reserve(int* first, int* second, long* n, int* null, int* small) {
    dbuf<double> b;
    const size_t huge = (size_t)1 << 50;
    *first = (int)b.reserve(huge);
    *second = (int)b.reserve(huge);
    *n = (long)b.n;
    *null = b.p == nullptr;
    cudaGetLastError();
    *small = (int)b.reserve(16);
}
"""


def test_reserve_after_a_failed_allocation():
    import paper_1007_5335_gb300  # noqa: F401  (the library itself)
    from native_access import compile_cuda
    lib = compile_cuda(SOURCE)
    first, second, null, small, n = ctypes.c_int(), ctypes.c_int(), ctypes.c_int(), ctypes.c_int(), ctypes.c_long()
    lib.failed_reserve(ctypes.byref(first), ctypes.byref(second), ctypes.byref(n), ctypes.byref(null),
                       ctypes.byref(small))
    assert first.value != 0 and second.value == first.value
    assert n.value == 0 and null.value == 1
    assert small.value == 0
