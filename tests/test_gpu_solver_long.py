"""The interactive GMRES over long lives and long bases: the counters that the host follows after 2^30
steps, bases on both sides of the cluster sizes' limit, and the form that keeps w in global memory.

The operator is replaced by a permutation with one cycle through node 0 (written into the boundary's dense
binary64 operator): from the unit vector of node 0 its Krylov basis is unit vectors, the residual stays 1
until the step that closes the cycle and is 0 there, so the solve takes exactly as many steps as the cycle
is long, its last step is a breakdown (w in the span), and the solution is a unit vector."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "gmres_kernels.cuh"
// (A x)_i = x_{i-1} on the nodes 0 .. m-1 (cyclic), x_i on the others
static __global__ void k_cycle(double* a, long n, long m) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i < n) a[i * n + (i < m ? (i + m - 1) % m : i)] = 1.0;
}
extern "C" int set_cycle(mh_boundary* b, long n, long m) {
    if (b->n != n || (long)b->op.A64.n < n * n || m > n) return -1;
    cudaMemset(b->op.A64.p, 0, n * n * 8);
    k_cycle<<<(unsigned)((n + 255) / 256), 256>>>(b->op.A64.p, n, m);
    return (int)cudaDeviceSynchronize();
}
extern "C" int set_matrix(mh_boundary* b, const double* a, long n) {
    if (b->n != n || (long)b->op.A64.n < n * n) return -1;
    return (int)cudaMemcpy(b->op.A64.p, a, n * n * 8, cudaMemcpyHostToDevice);
}
extern "C" int set_cluster(mh_boundary* b, int blocks) {
    const int had = b->ws.cluster;
    b->ws.cluster = blocks;
    return had;
}
extern "C" void set_steps(mh_boundary* b, int v) { static_cast<gmres_k::progress*>(b->ws.prog)->steps = v; }
"""


@pytest.fixture(scope="module")
def native():
    import paper_1007_5335_gb300  # noqa: F401  (the library itself)
    from native_access import compile_cuda
    lib = compile_cuda(SOURCE)
    lib.set_cycle.argtypes = [ctypes.c_void_p, ctypes.c_long, ctypes.c_long]
    lib.set_steps.argtypes = [ctypes.c_void_p, ctypes.c_int]
    lib.set_matrix.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long]
    lib.set_cluster.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return lib


def _boundary(n, alpha):
    import torch

    import mh_workloads as W
    import paper_1007_5335_gb300 as mh
    ctx = mh.Context(0)
    bnd = mh.Boundary(ctx, [W.circle_nodes((0.0, 0.0), 1.0, n, clockwise=False)], alpert_order=8)
    x = torch.zeros(n, dtype=torch.float64, device="cuda:0")
    mh.mh_double_layer_apply(ctx, bnd, alpha, x, torch.empty_like(x))   # assembles the operator
    return mh, ctx, bnd


@pytest.mark.parametrize("prec", [0, 1])
def test_counter_after_two_to_the_thirty_steps(native, prec):
    import torch
    n, alpha = 256, 0.05
    mh, ctx, bnd = _boundary(n, alpha)
    rhs = torch.tensor(np.random.default_rng(3).standard_normal(n), device="cuda:0")
    a, b = torch.zeros_like(rhs), torch.zeros_like(rhs)
    one = mh.mh_gmres_solve(ctx, bnd, alpha, rhs, a, tol=1e-11, max_iter=100, prec=prec)
    assert one.iterations > 4
    native.set_steps(bnd.h, 2 * (2 ** 30 - 3))
    two = mh.mh_gmres_solve(ctx, bnd, alpha, rhs, b, tol=1e-11, max_iter=100, prec=prec)
    assert two.converged and two.iterations == one.iterations
    assert torch.equal(a, b)


@pytest.mark.parametrize("n,cycle", [
    (30, 30),         # most blocks of the cluster hold no row
    (400, 400),       # 8 blocks
    (1030, 900),      # 16 blocks up to 400 vectors, then 8
    (24000, 995),     # the slice of w no longer fits in shared memory beside the sums of ~980 vectors
])
def test_cyclic_shift(native, n, cycle):
    import torch
    alpha = 0.3
    mh, ctx, bnd = _boundary(n, alpha)
    torch.cuda.synchronize()
    assert native.set_cycle(bnd.h, n, cycle) == 0
    rhs = torch.zeros(n, dtype=torch.float64, device="cuda:0")
    rhs[0] = 1.0
    x = torch.zeros_like(rhs)
    info = mh.mh_gmres_solve(ctx, bnd, alpha, rhs, x, tol=1e-12, max_iter=1000, prec=mh.MH_PREC_FP64)
    assert info.converged and info.iterations == cycle
    ref = torch.zeros_like(x)
    ref[cycle - 1] = 1.0                                           # A e_{m-1} = e_0
    assert (x - ref).abs().max().item() <= 1e-12


def _general(native, n, seed, cluster=None):
    """A solve with a full operator (standard normal entries / sqrt(n) + 1.2 I: eigenvalues in a disc that nearly
    reaches 0, so GMRES takes many steps) against the direct one: ||x - ref|| <= tol ||b|| ||A^-1||, plus the
    direct solve's own rounding."""
    import torch
    alpha = 0.3
    mh, ctx, bnd = _boundary(n, alpha)
    rng = np.random.default_rng(seed)
    A = np.ascontiguousarray(rng.standard_normal((n, n)) / np.sqrt(n) + 1.2 * np.eye(n))
    rhs = rng.standard_normal(n)
    torch.cuda.synchronize()
    assert native.set_matrix(bnd.h, A.ctypes.data, n) == 0
    x = torch.zeros(n, dtype=torch.float64, device="cuda:0")
    b = torch.tensor(rhs, device="cuda:0")
    if cluster:
        mh.mh_gmres_solve(ctx, bnd, alpha, b, x, tol=0.5, max_iter=1000)   # makes the workspace
        assert native.set_cluster(bnd.h, cluster) in (8, 16)
        x.zero_()
    info = mh.mh_gmres_solve(ctx, bnd, alpha, b, x, tol=1e-11, max_iter=1000, prec=mh.MH_PREC_FP64)
    ref = np.linalg.solve(A, rhs)
    inv = np.linalg.norm(np.linalg.inv(A), 2)
    bound = 1e-11 * np.linalg.norm(rhs) * inv + n * 2.3e-16 * np.linalg.cond(A) * np.linalg.norm(ref)
    assert np.linalg.norm(x.cpu().numpy() - ref) <= bound
    return info


@pytest.mark.parametrize("n", [40, 130, 600])
def test_long_triangular_solve(native, n):
    assert _general(native, n, n).iterations > 32


def test_cluster_of_eight_on_a_long_boundary(native):
    assert _general(native, 1100, 1, cluster=8).iterations > 32
