"""Binary64 evaluation at targets from two host threads, a context and a stream each, on one boundary:
every call gives what it gives alone.  Curves of 2^L nodes and others (the two forms of the fine weights),
targets of all regimes (normal line, upsampled, trapezoid) in sets of different sizes, so that the
calls also differ in the buffers they need.

Bound: a target's sum adds its curves' upsampled sums atomically, in either order: two roundings of the sum
of the absolute terms, taken as 1e-13 of the largest value."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [256, 288])
def test_two_threads_on_one_boundary(n):
    import torch

    import mh_workloads as W
    import paper_1007_5335_gb300 as mh

    alpha = 0.1
    curves = [W.circle_nodes((0.0, 0.0), 1.0, n, clockwise=False), W.circle_nodes((0.1, 0.0), 0.4, n, clockwise=True)]
    ctx = mh.Context(0)
    bnd = mh.Boundary(ctx, curves, alpert_order=8)
    rng = np.random.default_rng(n)
    jobs = []
    for k, m in enumerate((700, 90)):
        rad = np.concatenate([1.0 - 10.0 ** rng.uniform(-6, -0.6, m // 2), rng.uniform(0.55, 0.75, m - m // 2)])
        ang = rng.uniform(0, 2 * np.pi, m)
        xy = torch.tensor(np.stack([rad * np.cos(ang), rad * np.sin(ang)], 1), device="cuda:0")
        sig = torch.tensor(rng.standard_normal(bnd.n) * 10.0 ** k, device="cuda:0")
        ref = torch.empty(m, dtype=torch.float64, device="cuda:0")
        mh.mh_double_layer_apply(ctx, bnd, alpha, sig, ref, xy, mh.MH_PREC_FP64)
        jobs.append((xy, sig, ref))
    torch.cuda.synchronize()
    worst, errors = [0.0, 0.0], []

    def work(k):
        try:
            xy, sig, ref = jobs[k]
            with torch.cuda.stream(torch.cuda.Stream()):
                own = mh.Context(0)
                out = torch.empty_like(ref)
                for _ in range(200):
                    mh.mh_double_layer_apply(own, bnd, alpha, sig, out, xy, mh.MH_PREC_FP64)
                    worst[k] = max(worst[k], ((out - ref).abs().max() / ref.abs().max()).item())
        except Exception as e:   # handed to the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert max(worst) <= 1e-13, worst
