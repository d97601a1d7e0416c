"""The binary64 pair term from its table (csrc/pair64.cuh) against K1 itself: the double layer at
targets in the trapezoid regime, where it is a plain sum over the nodes.  alpha^2 sits on, just
below and just above a power of two (the table's octaves start at powers of two) and the distances
run from a few node spacings to beyond the cut at 45 alpha; odd target counts cross the kernel's
tiles.

Bound: a pair's r^2 carries two roundings, so K1(z) moves by (z/2 + 1) 2 eps, at most 1e-14 for
z <= 45; the polynomial, the products and scipy's K1 add a few eps: 2e-14 of the sum of the
absolute terms."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha2", [2.0 ** -10, np.nextafter(2.0 ** -10, 0), np.nextafter(2.0 ** -10, 1), 1e-4, 0.03, 4.0])
@pytest.mark.parametrize("n_targets", [1, 129])
def test_pair_table_against_k1(alpha2, n_targets):
    import torch
    from scipy.special import k1

    import mh_workloads as W
    import paper_1007_5335_gb300 as mh

    n = 640
    alpha = math.sqrt(float(alpha2))
    curve = W.circle_nodes((0.0, 0.0), 1.0, n, clockwise=False)
    ctx = mh.Context(0)
    bnd = mh.Boundary(ctx, [curve], alpert_order=8)
    rng = np.random.default_rng(n_targets)
    rad = rng.uniform(0.0, 1.0 - 12 * 2 * math.pi / n, n_targets)   # farther than 10 node spacings
    ang = rng.uniform(0.0, 2 * math.pi, n_targets)
    xy = np.stack([rad * np.cos(ang), rad * np.sin(ang)], axis=1)
    sigma = rng.standard_normal(n)
    out = torch.empty(n_targets, dtype=torch.float64, device="cuda:0")
    mh.mh_double_layer_apply(ctx, bnd, alpha, torch.tensor(sigma, device="cuda:0"), out,
                             torch.tensor(xy, device="cuda:0"), mh.MH_PREC_FP64)
    d = curve[None] - xy[:, None]
    r = np.hypot(d[..., 0], d[..., 1])
    terms = -k1(r / alpha) / alpha * (d * curve[None]).sum(-1) / r * sigma * (2 * math.pi / n) / (2 * math.pi * alpha ** 2)
    terms[r > 45 * alpha] = 0.0
    err = np.abs(out.cpu().numpy() - terms.sum(1))
    # pairs at the cut itself may fall on either side of it: below e^-45 of the largest term each
    edge = np.exp(-45.0) * n / alpha ** 3
    assert np.all(err <= 2e-14 * np.abs(terms).sum(1) + edge), (err / np.abs(terms).sum(1)).max()
