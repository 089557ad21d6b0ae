"""Launch configurations on requests that the warp-specialised kernel takes (the small ones of the other
tuning tests run on the band kernel), and tuning on requests that it does not."""
import pytest

from graph_util import captured

pytestmark = pytest.mark.gpu


def _plan(kappa, n_theta, n_phi, H, flags=0):
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, Plan
    return Plan(list(kappa), 1.0, n_theta, n_phi, flags=flags | (0 if H else SMERF_ORDER_PAPER), anchor_spacing=H)


def _kernel(plan, n):
    import torch
    out = torch.empty(n, plan.n_theta, plan.n_phi, dtype=plan.dtype, device="cuda")
    return captured(lambda: plan.sample(1, n, out=out))[0][-1]


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("kappa,n_theta,n_phi,H,n", [((20.0, 50.0), 20, 512, 4, 131), ((30.0,), 10, 4096, 4, 81),
                                                   ((10.0,), 8, 256, 0, 801), ((10.0, 20.0, 40.0), 10, 1024, 4, 81)])
def test_every_candidate_gives_the_same_field_on_the_warp_specialised_kernel(fp64, kappa, n_theta, n_phi, H, n):
    import torch
    from paper_1709_10314_gb300 import SMERF_RECUR_FP64
    plan = _plan(kappa, n_theta, n_phi, H, SMERF_RECUR_FP64 if fp64 else 0)
    ref, first = plan.sample(7, n), {}
    for cfg in plan.launch_candidates():
        plan.set_launch(cfg)
        name = _kernel(plan, n)
        assert "segment_ws_kernel" in name and "Li%dELi%dELi%dELi%dE" % (len(kappa), cfg[0], cfg[1], cfg[4]) in name
        got = plan.sample(7, n)
        assert torch.equal(got, first.setdefault(cfg[5], got)), cfg
    assert torch.equal(ref, first[16] if 16 in first else first[4])


@pytest.mark.parametrize("kappa,n_theta,n_phi,H", [((20.0, 50.0), 48, 512, 16), ((30.0,), 64, 1024, 8), ((10.0,), 32, 64, 0),
                                                  ((6.0, 11.0, 25.0), 32, 64, 4), ((20.0,), 24, 2048, 0), ((20.0, 50.0), 40, 2048, 8)])
@pytest.mark.parametrize("fp64", [False, True])
def test_tuning_on_a_band_kernel_request_keeps_the_built_in_choice(kappa, n_theta, n_phi, H, fp64):
    from paper_1709_10314_gb300 import SMERF_RECUR_FP64
    flags = SMERF_RECUR_FP64 if fp64 else 0
    plan, fresh = _plan(kappa, n_theta, n_phi, H, flags), _plan(kappa, n_theta, n_phi, H, flags)
    assert "segment_band_kernel" in _kernel(plan, 1)
    chosen = plan.autotune(1)
    assert tuple(chosen) in [tuple(c) for c in plan.launch_candidates()]
    for n in (1, 64, 2000 if n_phi < 512 else 200):
        assert _kernel(plan, n) == _kernel(fresh, n)


def test_tuning_a_ring_plan_takes_a_configuration_with_a_ring_build():
    import torch
    plan = _plan((20.0,), 40, 4096, 8)
    plan.set_rings([4096] * 40)
    ref = plan.sample(3, 16)
    chosen = plan.autotune(16)
    assert tuple(chosen) in [tuple(c) for c in plan.launch_candidates()]
    out = torch.empty_like(ref)
    assert "segment_ws_kernel" in captured(lambda: plan.sample(3, 16, out=out))[0][-1]
    if chosen[5] == 16:
        assert torch.equal(plan.sample(3, 16), ref)


def test_a_batch_group_takes_the_launch_of_its_size():
    """p = 3 requests of one shape: few of them the launch of as many segments of a single call (large CTAs, one
    wave), many the throughput launch; the same fields."""
    import re
    import torch
    from paper_1709_10314_gb300 import Batch
    plans = [_plan((10.0 + 0.3 * i, 20.0, 40.0), 64, 2048, 4) for i in range(24)]

    def run(plans, counts):
        b = Batch(plans, counts)
        outs = [torch.full((n, p.n_theta, p.n_phi), float("nan"), device="cuda") for p, n in zip(plans, counts)]
        b.sample(list(range(len(plans))), outs)
        for i, (p, n, o) in enumerate(zip(plans, counts, outs)):
            assert torch.equal(o, p.sample(i, n))
        name = captured(b.launch)[0][-1]
        b.close()
        return re.search(r"Li3ELi(\d)ELi1ELi1E", name).group(1)

    upt = lambda n: re.search(r"Li3ELi(\d)ELi1ELi1E", _kernel(plans[0], n)).group(1)  # noqa: E731
    few, many = run(plans[:2], [1, 1]), run(plans, [3] * 24)
    assert few == upt(2) and many == upt(72) and few != many
