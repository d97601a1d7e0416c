"""Classification of targets in domains of any size: a geometry scaled by a power of two has the same
classes, and U^h scales by alpha^-2 (every length in the kernel appears relative to alpha).

Scaling by a power of two changes no rounding, except where a bound of the number range is met; the sums of
several curves are added atomically, in either order: 1e-13 of the largest value.

And holes of 1e-8 of the domain, which binary32 positions do not resolve: one around a volume node, one
beside another node (two radii from its edge)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("e", [-60, -40, 40, 70])
def test_scaled_domain(e):
    import torch

    import mh_workloads as W
    import paper_1007_5335_gb300 as mh

    n = 256
    base = [W.circle_nodes((0.0, 0.0), 1.0, n, clockwise=False), W.circle_nodes((0.2, 0.0), 0.3, n, clockwise=True)]
    rng = np.random.default_rng(0)
    rad = 1.0 - 10.0 ** rng.uniform(-5, -0.2, 400)
    ang = rng.uniform(0, 2 * np.pi, 400)
    xy = np.stack([rad * np.cos(ang), rad * np.sin(ang)], 1)
    xy = xy[np.hypot(xy[:, 0] - 0.2, xy[:, 1]) > 0.31]
    sig = torch.tensor(rng.standard_normal(2 * n), device="cuda:0")

    def run(s):
        ctx = mh.Context(0)
        bnd = mh.Boundary(ctx, [c * s for c in base], alpert_order=8)
        tree = mh.Tree(ctx, (-1.25 * s, -1.25 * s, 2.5 * s), 4, 3, 3)
        prob = mh.Problem(ctx, tree, bnd, (0.25 * s) ** 2, 8, ext_mode=mh.MH_EXT_CONST, ext_const=[0.0, 0.0])
        out = torch.empty(len(xy), dtype=torch.float64, device="cuda:0")
        mh.mh_double_layer_apply(ctx, bnd, 0.25 * s, sig, out, torch.tensor(xy * s, device="cuda:0"), mh.MH_PREC_FP64)
        return prob.regions(), out.cpu().numpy() * s * s

    reg0, u0 = run(1.0)
    assert set(reg0) == {-1, 0, 1}
    reg, u = run(2.0 ** e)
    assert np.array_equal(reg, reg0)
    assert np.max(np.abs(u - u0)) <= 1e-13 * np.max(np.abs(u0))


def test_holes_below_binary32_resolution():
    import mh_workloads as W
    import paper_1007_5335_gb300 as mh

    ctx = mh.Context(0)
    tree = mh.Tree(ctx, (-1.25, -1.25, 2.5), 4, 3, 3)
    nodes = tree.nodes().cpu().numpy()
    i = int(np.argmin(np.hypot(nodes[:, 0] - 0.5, nodes[:, 1] - 0.3)))
    j = int(np.argmin(np.hypot(nodes[:, 0] + 0.4, nodes[:, 1] + 0.2)))
    r, n = 1e-8, 256
    curves = [W.circle_nodes((0.0, 0.0), 1.0, n, clockwise=False),
              W.circle_nodes(tuple(nodes[i]), r, n, clockwise=True),
              W.circle_nodes((nodes[j, 0] + 3 * r, nodes[j, 1]), r, n, clockwise=True)]
    bnd = mh.Boundary(ctx, curves, alpert_order=8)
    prob = mh.Problem(ctx, tree, bnd, 0.01, 8, ext_mode=mh.MH_EXT_CONST, ext_const=[0.0] * 3)
    ref = np.where(np.hypot(nodes[:, 0], nodes[:, 1]) < 1.0, -1, 0)
    ref[i] = 1
    assert np.array_equal(prob.regions(), ref)
