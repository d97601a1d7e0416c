"""The tabulated pair factor f(rho) = K1(z)/z (csrc/pair64.cuh) against a reference of more digits: the
trapezoid sum of K1(z) e^z = int_0^oo exp(-2 z sinh^2(t/2)) cosh t dt in extended precision, whose error falls
like exp(-pi^2/h) (h = 1/16: far below binary64), checked against K1's expansion where it is simple.

Bound, in units of 2^-53: K1 at a centre 5 (a series of three terms of either sign below z = 2; exp, rsqrt
and a Clenshaw sum above), its division 1, the last product and sum 2, plus the first term left out and the
binary32 rounding of the terms tau^4..6, both at their largest (bin edges): 4.2e-16 + 2.4e-16 up to z = 8,
1e-15 + 8e-16 beyond, reached at the cut only, where they grow like z^7 and z^4."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "mh_internal.cuh"
#include "pair64.cuh"
static __global__ void k_eval(mh_pair_tab T, const double* rho, long n, double* out) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i < n) out[i] = mh_pair_f(rho[i], T);
}
extern "C" int pair_f(double alpha, const double* rho, long n, double* out) {
    dbuf<double2> t;
    dbuf<double> r, o;
    if (t.alloc(PT_WORDS * PT_BINS) || r.alloc(n) || o.alloc(n)) return -1;
    cudaMemcpy(r.p, rho, n * 8, cudaMemcpyHostToDevice);
    k_pair_table<<<(PT_BINS + 127) / 128, 128>>>(mh_pair_tab_make(nullptr, alpha), alpha, t.p);
    k_eval<<<(unsigned)((n + 255) / 256), 256>>>(mh_pair_tab_make(t.p, alpha), r.p, n, o.p);
    return (int)cudaMemcpy(out, o.p, n * 8, cudaMemcpyDeviceToHost);
}
"""


def _k1_over_z(z):
    """K1(z)/z in np.longdouble."""
    L = np.longdouble
    h = L(1) / L(16)
    total = np.full(z.shape, L(0.5))                     # t = 0
    for k in range(1, 400):
        t = h * k
        s = np.sinh(t / 2)
        term = np.exp(-2 * z * s * s) * np.cosh(t)
        total = total + term
        if np.all(term < 1e-25 * total):
            break
    return total * h * np.exp(-z) / z


@pytest.mark.parametrize("alpha2", [1e-3, 2.0 ** -10, 0.03, 7.0])
def test_pair_factor(alpha2):
    import paper_1007_5335_gb300  # noqa: F401  (the library itself)
    from native_access import compile_cuda
    if np.finfo(np.longdouble).eps > 1.1e-19:
        pytest.skip("no extended precision on this machine")
    L = np.longdouble
    lib = compile_cuda(SOURCE)
    lib.pair_f.argtypes = [ctypes.c_double, ctypes.c_void_p, ctypes.c_long, ctypes.c_void_p]
    alpha = float(np.sqrt(alpha2))
    rng = np.random.default_rng(5)
    z = np.concatenate([np.exp(rng.uniform(np.log(1 / 127), np.log(44.9), 3000)), rng.uniform(2, 44.9, 3000)])
    rho = np.ascontiguousarray((z * alpha) ** 2)
    out = np.empty_like(rho)
    assert lib.pair_f(alpha, rho.ctypes.data, rho.size, out.ctypes.data) == 0
    zl = np.sqrt(L(1) * rho) / L(alpha)
    ref = _k1_over_z(zl)
    err = np.abs((out - ref) / ref).astype(np.float64)
    zf = zl.astype(np.float64)
    bound = 8 * 2.0 ** -53 + np.where(zf <= 8, 6.6e-16, 1e-15 * (zf / 45) ** 7 + 8e-16 * (zf / 45) ** 4)
    assert np.all(err <= bound), (err / bound).max()
