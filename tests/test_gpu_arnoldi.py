"""The cluster form of the Arnoldi step (csrc/gmres_kernels.cuh) where its slices, tiles and
cluster sizes change: the smallest boundary (most blocks of the cluster hold no row), ragged slices,
both cluster sizes, and bases longer than the block's warps.

Against a direct solve with the same operator (its columns from products with unit vectors).  The
returned density has ||b - A x|| <= tol ||b||, so ||x - x_ref|| <= tol ||b|| ||A^-1||, plus the
direct solve's own rounding (n eps cond)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _curves(n, holes):
    import mh_workloads as W
    out = [W.circle_nodes((0.0, 0.0), 1.0, n, clockwise=False)]
    for j in range(holes):
        c = (0.5 * math.cos(2.1 * j), 0.5 * math.sin(2.1 * j))
        out.append(W.starfish_nodes(c, 0.15, 0.3, 5, n, clockwise=True))
    return out


@pytest.mark.parametrize("n,holes,alpha", [(20, 0, 0.3), (30, 1, 0.2), (254, 0, 0.05), (342, 2, 1.0), (512, 1, 0.1),
                                           (350, 2, 2.0)])
@pytest.mark.parametrize("prec", [0, 1])
def test_solve_against_direct(n, holes, alpha, prec):
    import torch

    import paper_1007_5335_gb300 as mh

    ctx = mh.Context(0)
    bnd = mh.Boundary(ctx, _curves(n, holes), alpert_order=8)
    m = bnd.n
    eye = torch.eye(m, dtype=torch.float64, device="cuda:0")
    A = torch.empty_like(eye)
    for j in range(m):
        mh.mh_double_layer_apply(ctx, bnd, alpha, eye[j], A[j])
    A = A.cpu().numpy().T
    rhs = np.random.default_rng(n).standard_normal(m)
    x = torch.zeros(m, dtype=torch.float64, device="cuda:0")
    tol = 1e-11
    info = mh.mh_gmres_solve(ctx, bnd, alpha, torch.tensor(rhs, device="cuda:0"), x, tol=tol, max_iter=200, prec=prec)
    ref = np.linalg.solve(A, rhs)
    inv = np.linalg.norm(np.linalg.inv(A), 2)
    bound = tol * np.linalg.norm(rhs) * inv + m * 2.3e-16 * np.linalg.cond(A) * np.linalg.norm(ref)
    assert np.linalg.norm(x.cpu().numpy() - ref) <= bound
    assert info.converged and info.rel_residual <= tol
