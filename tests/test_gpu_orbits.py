"""Binary64 contractions by reflection orbits (csrc/orbit.cuh) where their sizes change: odd and even
numbers of nodes a side (a middle node is its own image), orders with empty classes (p = 1), the
largest operators of one block, uniform and adaptive trees (M2P, P2L, neighbours of other sizes).

Against the plain contractions in binary32 on the CUDA cores, operator by operator: passes of up to
121 products each, 2^-24 a product, six passes in a row: 121 * 6 * 6e-8 = 4.4e-5 of the largest value.
A wrong sign or a wrong image is an error of the order of a neighbour's contribution."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("adaptive", [False, True])
@pytest.mark.parametrize("q,p", [(2, 1), (3, 2), (4, 20), (5, 7), (8, 20), (8, 40), (11, 12)])
def test_orbits(q, p, adaptive):
    import torch

    import paper_1007_5335_gb300 as mh

    ctx = mh.Context(0)
    if adaptive:
        def forcing(xy):
            return np.exp(-80.0 * ((xy[:, 0] - 0.3) ** 2 + (xy[:, 1] + 0.2) ** 2))

        tree = mh.Tree(ctx, (-1.0, -1.0, 2.0), q, 2, 5, forcing, {2: 3e-2, 3: 1e-2}.get(q, 1e-5))
    else:
        tree = mh.Tree(ctx, (-1.0, -1.0, 2.0), q, 3, 3)
    b = torch.tensor(np.random.default_rng(q + p).standard_normal(tree.n_nodes), device="cuda:0")
    u, plain = torch.empty_like(b), torch.empty_like(b)
    mh.mh_volume_potential(ctx, tree, 0.4, p, b, u)
    ctx.tensor_cores(False)
    mh.mh_volume_potential(ctx, tree, 0.4, p, b, plain, prec=mh.MH_PREC_MIXED)
    assert float((u - plain).abs().max() / u.abs().max()) <= 4.4e-5
