"""The band kernel's early start: it reads its step tables before it waits for the launch before it,
so that launch must not be the one that writes them (FP64 tables converted to FP32 per call)."""
import pytest

from graph_util import captured

pytestmark = pytest.mark.gpu


def _plan(kappa, n_theta, n_phi, H, tables64):
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, SMERF_TABLES_FP32, SMERF_TABLES_FP64, Plan
    flags = (SMERF_TABLES_FP64 if tables64 else SMERF_TABLES_FP32) | (0 if H else SMERF_ORDER_PAPER)
    return Plan(kappa, 1.0, n_theta, n_phi, flags=flags, anchor_spacing=H)


@pytest.mark.parametrize("n_theta,n_phi,H,tables64,n,anchors,early", [
    (100, 512, 0, True, 4, "anchor_stage_kernel", False),   # Alg. 2's order
    (100, 256, 16, True, 8, "anchor_stage_kernel", False),  # three anchors per chain
    (40, 128, 4, True, 4, "anchor_tile_kernel", True),      # the tables are ready before the anchors start
    (100, 512, 0, True, 3, "anchor_kernel", True),          # no conversion
    (100, 512, 0, False, 4, "anchor_kernel", True),
])
def test_no_early_start_behind_the_launch_that_writes_the_tables(n_theta, n_phi, H, tables64, n, anchors, early):
    import torch
    plan = _plan([6.0, 15.0], n_theta, n_phi, H, tables64)
    out = torch.empty(n, n_theta, n_phi, device="cuda")
    kernels, edges = captured(lambda: plan.sample(3, n, out=out))
    assert anchors in kernels[-2] and "segment_band_kernel" in kernels[-1]
    assert edges == ([(kernels[-2], kernels[-1])] if early else [])


@pytest.mark.parametrize("n_theta,n_phi,H,n", [(100, 512, 0, 4), (100, 256, 16, 8), (34, 2048, 16, 40)])
def test_plans_in_turn_on_one_stream(n_theta, n_phi, H, n):
    """Two plans' calls in turn, whose converted tables take the same memory: each field is that of the
    same realisations drawn one by one (which convert nothing)."""
    import torch
    plans = [_plan([6.0, 15.0], n_theta, n_phi, H, True), _plan([60.0, 150.0], n_theta, n_phi, H, True)]
    ref = [torch.cat([p.sample(20 + r, 1) for r in range(n)]) for p in plans]
    outs = [torch.empty_like(ref[0]) for _ in range(2)]
    for _ in range(40):
        for p, o in zip(plans, outs):
            o.zero_()
            p.sample(20, n, out=o)
        assert torch.equal(outs[0], ref[0]) and torch.equal(outs[1], ref[1])


@pytest.mark.parametrize("p,n_theta,n_phi,H,n,fp64,tables64", [
    (1, 64, 128, 0, 1, True, False),
    (2, 181, 512, 16, 1, False, False),
    (2, 40, 128, 4, 4, False, True),     # tables converted ahead of the tiles
    (2, 100, 512, 0, 4, False, True),    # tables converted beside the anchors: no early start
    (2, 32, 64, 0, 1200, True, False),   # two realisations per CTA
])
def test_small_requests_captured_and_replayed(p, n_theta, n_phi, H, n, fp64, tables64):
    """A captured small request (an early start is a programmatic edge of the graph) gives the call's field at
    every replay, alone and between other work on the stream."""
    import torch
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, SMERF_RECUR_FP64, SMERF_TABLES_FP64, Plan
    flags = (SMERF_RECUR_FP64 if fp64 else 0) | (SMERF_TABLES_FP64 if tables64 else 0) | (0 if H else SMERF_ORDER_PAPER)
    plan = Plan([6.0, 15.0][:p], 1.0, n_theta, n_phi, flags=flags, anchor_spacing=H)
    ref = plan.sample(9, n)
    out, s, g = torch.empty_like(ref), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        plan.sample(9, n, out=out)  # the first launch outside the capture
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        plan.sample(9, n, out=out)
    for other in (False, True, True):
        out.zero_()
        torch.cuda.synchronize()
        if other:
            plan.sample(10, n, out=torch.empty_like(out))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
