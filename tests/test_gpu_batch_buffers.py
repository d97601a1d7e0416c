"""Buffers that a recorded batch graph holds: work of the other precision on the same problem between
two batch steps must not replace them.

The shares of the auxiliary trapezoid sums differ between the precisions (whole tiles of 128 sources in
binary32, multiples of 16 in binary64), so do their partial sums.  The sequence first makes everything
else a binary64 step would create (Krylov workspace, pair table), so that nothing but the partial sums
could force a new recording."""
import pytest

import mh_workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_binary64_step_between_mixed_batch_steps():
    import paper_1007_5335_gb300 as mh
    ctx = mh.Context(0)
    wl = W.batch_problem(0, npc=256, refine_tol=1e-5)

    def make():
        tree = mh.Tree(ctx, wl.box, wl.q, wl.min_level, wl.max_level, wl.forcing, wl.refine_tol)
        bnd = mh.Boundary(ctx, wl.curves, alpert_order=8)
        prob = mh.Problem(ctx, tree, bnd, wl.dt, 16, ext_mode=mh.MH_EXT_CONST, ext_const=wl.ext_const)
        F = torch.tensor(wl.forcing(tree.nodes().cpu().numpy()), device="cuda")
        z = lambda n: torch.zeros(n, dtype=torch.float64, device="cuda")
        return dict(tree=tree, bnd=bnd, prob=prob, F=F, f=z(bnd.n), u=z(tree.n_nodes), s=z(bnd.n), t=z(tree.n_nodes))

    def single(p, prec):
        mh.heat_step(ctx, p["prob"], p["u"], p["F"], p["f"], p["t"], p["s"], gmres_tol=1e-10, prec=prec)
        p["u"].copy_(p["t"])

    a, b = make(), make()
    batch = mh.Batch(ctx, [a["prob"]])

    def batched():
        batch.step([a["u"]], [a["F"]], [a["f"]], [a["s"]], gmres_tol=1e-10, prec=mh.MH_PREC_MIXED)

    # Krylov workspace and the pair table of this alpha
    single(a, mh.MH_PREC_MIXED), single(b, mh.MH_PREC_MIXED)
    pts = torch.tensor(a["tree"].nodes().cpu().numpy()[a["prob"].regions() == -1][:64], device="cuda")
    mh.mh_double_layer_apply(ctx, a["bnd"], wl.dt ** 0.5, a["s"], torch.empty(64, dtype=torch.float64, device="cuda"), pts)
    batched(), single(b, mh.MH_PREC_MIXED)          # records the graph
    batched(), single(b, mh.MH_PREC_MIXED)          # replays it
    torch.cuda.synchronize()
    before = mh.device_alloc_calls()
    single(a, mh.MH_PREC_FP64)
    # at most the pair table is made here (one allocation); a replaced buffer counts twice, a free and an allocation
    assert mh.device_alloc_calls() - before <= 1, "a step replaced a buffer that the recorded graph may hold"
    single(b, mh.MH_PREC_FP64)
    for _ in range(2):
        batched(), single(b, mh.MH_PREC_MIXED)
    ins = torch.tensor(b["prob"].regions() == -1, device="cuda")
    # both solvers stop at 1e-10 of the right-hand side; the binary32 passes differ by their rounding (1e-7)
    assert (torch.linalg.norm((a["u"] - b["u"])[ins]) / torch.linalg.norm(b["u"][ins])).item() <= 1e-7
