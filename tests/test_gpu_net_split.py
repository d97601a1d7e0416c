"""Training products split over k (csrc/net.cu k_gemm) at the sizes where tiles, slabs and splits
change: one sample, ragged tiles, widths from the smallest, k below and far above a slab, and two
calls in a row (the tile counters reset themselves).

Loss and gradient against the same network in binary64 torch.  A binary32 dot product of length k
with random signs is off by about sqrt(k) eps; 8 products in a row and a factor 4: the gradient's
relative 2-norm error is at most 32 sqrt(k_max) 2^-24."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,curves,modes,width,rows", [(32, 1, 4, 8, 1), (64, 2, 32, 72, 5), (256, 3, 100, 64, 65),
                                                           (512, 2, 256, 256, 64), (128, 1, 64, 200, 300)])
def test_loss_and_gradient(nodes, curves, modes, width, rows):
    import torch

    import mh_workloads as W
    import paper_1007_5335_gb300 as mh

    cs = [W.circle_nodes((0.0, 0.0), 1.0, nodes, clockwise=False)]
    cs += [W.circle_nodes((0.4 * math.cos(2 * j), 0.4 * math.sin(2 * j)), 0.1, nodes, clockwise=True) for j in range(curves - 1)]
    ctx = mh.Context(0)
    net = mh.Net(ctx, mh.Boundary(ctx, cs, alpert_order=8), modes, width)
    rng = np.random.default_rng(rows)
    d = net.d
    par = []
    for o, i in ((width, d), (width, width), (width, width), (d, width)):
        par += [(rng.standard_normal((o, i)) / math.sqrt(i)).astype(np.float32), (0.1 * rng.standard_normal(o)).astype(np.float32)]
    net.set_params(np.concatenate([a.reshape(-1) for a in par]))
    X, T = (torch.tensor(rng.standard_normal((rows, d)).astype(np.float32), device="cuda:0") for _ in range(2))
    g = torch.empty(net.n_params, dtype=torch.float32, device="cuda:0")
    for _ in range(2):
        loss = net.loss_grad(X, T, g)
        p64 = [torch.tensor(a, device="cuda:0").double().requires_grad_() for a in par]
        h = X.double()
        for l in range(4):
            h = h @ p64[2 * l].T + p64[2 * l + 1]
            h = torch.tanh(h) if l < 3 else h
        ref = (h - T.double()).square().mean() / 2
        ref.backward()
        gr = torch.cat([a.grad.reshape(-1) for a in p64])
        tol = 32 * math.sqrt(max(d, width, rows)) * 2.0 ** -24
        assert abs(loss - float(ref.detach())) <= tol * float(ref.detach())
        assert float((g.double() - gr).norm() / gr.norm()) <= tol
        g.zero_()
