"""Outputs formed from single columns (csrc/volume.cu k_cols) where their sizes change: leaves whose
sources fill several chunks of 256 columns, leaves with a few, ragged groups of 16 boundary nodes,
and a second product (the counters of cut outputs reset themselves).

The matrix-free operator against the stored one.  The multipole series of well separated boxes
converges at least like 0.55^n: 4e-11 of the far field at p = 40, plus rounding: 1e-9 of the
product's 2-norm."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npc,holes,level", [(2400, 0, 2), (1100, 1, 2), (126, 1, 3), (300, 2, 4)])
def test_columns(npc, holes, level):
    import torch

    import mh_workloads as W
    import paper_1007_5335_gb300 as mh

    cs = [W.circle_nodes((0.0, 0.0), 0.9, npc, clockwise=False)]
    cs += [W.starfish_nodes((0.5 * math.cos(2.5 * j), 0.5 * math.sin(2.5 * j)), 0.15, 0.3, 5, npc, clockwise=True)
           for j in range(holes)]
    ctx = mh.Context(0)
    tree = mh.Tree(ctx, (-1.0, -1.0, 2.0), 4, level, level)
    bnd = mh.Boundary(ctx, cs, alpert_order=8)
    prob = mh.Problem(ctx, tree, bnd, 0.01, 40)
    rng = np.random.default_rng(npc)
    xs = [torch.tensor(rng.standard_normal(bnd.n), device="cuda:0") for _ in range(2)]
    dense = [mh.mh_double_layer_apply(ctx, bnd, prob.alpha, x, torch.empty_like(x)) for x in xs]
    prob.matrix_free(True)
    for x, ref in zip(xs, dense):
        y = mh.mh_double_layer_apply(ctx, bnd, prob.alpha, x, torch.empty_like(x))
        assert float((y - ref).norm() / ref.norm()) <= 1e-9
