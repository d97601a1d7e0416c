"""Entry points behind a caller's kernels that use programmatic dependent launch in their own way.

The caller's first kernel releases its dependents at once and writes its output a millisecond later (a bounded
delay); its second one is such a dependent that never waits, so it ends while the first still runs.  A call that
started as a dependent of the second would read the input before it is written.  Every entry point
therefore starts with an ordinary launch: the result is that of the call alone, bit for bit."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
static __global__ void k_late_copy(const char* src, char* dst, long bytes) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long t0 = clock64();
    for (int i = 0; i < 1000000 && clock64() - t0 < 2000000; ++i) {}
    for (long e = threadIdx.x; e < bytes; e += blockDim.x) dst[e] = src[e];
}
static __global__ void k_no_wait() {}
extern "C" int late_copy(const char* src, char* dst, long bytes, cudaStream_t st) {
    k_late_copy<<<1, 256, 0, st>>>(src, dst, bytes);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(32);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, k_no_wait);
}
"""


@pytest.fixture(scope="module")
def world():
    import torch

    import mh_workloads as W
    import paper_1007_5335_gb300 as mh
    from native_access import compile_cuda
    lib = compile_cuda(SOURCE, link_lib=False)
    lib.late_copy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long, ctypes.c_void_p]

    def late(src, dst):
        assert src.numel() == dst.numel() and src.dtype == dst.dtype
        assert lib.late_copy(src.data_ptr(), dst.data_ptr(), src.numel() * src.element_size(),
                             torch.cuda.current_stream().cuda_stream) == 0

    n = 512
    ctx = mh.Context(0)
    bnd = mh.Boundary(ctx, [W.circle_nodes((0.0, 0.0), 1.0, n, clockwise=False)], alpert_order=8)
    tree = mh.Tree(ctx, (-1.25, -1.25, 2.5), 8, 3, 3)
    return dict(mh=mh, W=W, torch=torch, late=late, ctx=ctx, bnd=bnd, tree=tree, n=n)


def _calls(w):
    """name -> (input, function of the input returning its outputs)"""
    mh, torch, ctx, bnd, tree, n = (w[k] for k in ("mh", "torch", "ctx", "bnd", "tree", "n"))
    rng = np.random.default_rng(1)
    dev = lambda a: torch.tensor(a, device="cuda:0")
    vec = dev(rng.standard_normal(n))
    nodes = dev(rng.standard_normal(tree.n_nodes))
    alpha = 0.2

    def product(prec):
        def f(x):
            y = torch.empty_like(x)
            mh.mh_double_layer_apply(ctx, bnd, alpha, x, y, prec=prec)
            return y
        return f

    def volume(prec):
        def f(b):
            u = torch.empty_like(b)
            mh.mh_volume_potential(ctx, tree, alpha, 12, b, u, prec)
            return u
        return f

    net = mh.Net(ctx, bnd, n_modes=32, width=32)
    net.set_params(0.1 * rng.standard_normal(net.n_params))
    X = dev(rng.standard_normal((16, net.d)).astype(np.float32))
    T = dev(rng.standard_normal((16, net.d)).astype(np.float32))

    def grad(x):
        g = torch.empty(net.n_params, dtype=torch.float32, device="cuda:0")
        net.loss_grad(x, T, g)
        return g

    def warm(x):
        x0, r0 = torch.empty_like(x), torch.empty_like(x)
        mh.mh_warm_start(ctx, bnd, alpha, mh.MH_WARM_PREVIOUS, x, vec, x0, r0)
        return r0

    return {"product_f64": (vec, product(0)), "product_mixed": (vec, product(1)),
            "volume_f64": (nodes, volume(0)), "volume_mixed": (nodes, volume(1)), "net_grad": (X, grad),
            "warm_start": (vec, warm)}


@pytest.mark.parametrize("name", ["product_f64", "product_mixed", "volume_f64", "volume_mixed", "net_grad", "warm_start"])
def test_behind_a_caller_that_does_not_wait(world, name):
    torch = world["torch"]
    x, call = _calls(world)[name]
    call(x)
    ref = call(x).clone()
    for _ in range(3):
        late_x = torch.zeros_like(x)
        torch.cuda.synchronize()
        world["late"](x, late_x)
        got = call(late_x)
        torch.cuda.synchronize()
        assert torch.equal(got, ref)


@pytest.mark.parametrize("prec", [0, 1])
def test_solve_behind_a_caller_that_does_not_wait(world, prec):
    mh, torch, n = world["mh"], world["torch"], world["n"]
    rng = np.random.default_rng(2)
    rhs, start = (torch.tensor(rng.standard_normal(n), device="cuda:0") for _ in range(2))

    def solve(x):
        mh.mh_gmres_solve(world["ctx"], world["bnd"], 0.2, rhs, x, tol=1e-9, max_iter=60, prec=prec)
        return x

    ref = solve(start.clone())
    for _ in range(3):
        x = torch.zeros_like(start)
        torch.cuda.synchronize()
        world["late"](start, x)
        assert torch.equal(solve(x), ref)
