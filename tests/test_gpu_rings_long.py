"""Ring-dependent longitudes on long rings, against the same plan's whole rings: their coefficients
evaluated at the rings' own points in FP64."""
import numpy as np
import pytest

from gpu_util import rel_err

pytestmark = pytest.mark.gpu


def _points(c, phi):
    """oracle.ring_values at given longitudes, the Nyquist coefficient's real part at any of them."""
    import torch
    c, phi = torch.as_tensor(c).cuda(), torch.as_tensor(phi).cuda()
    M = len(c) - 1
    t = torch.outer(phi, torch.arange(1, M, device="cuda", dtype=torch.float64))
    v = c[0].real + 2.0 * (torch.cos(t) @ c[1:M].real - torch.sin(t) @ c[1:M].imag)
    return (v + c[M].real * torch.cos(M * phi)).cpu().numpy()


def _worst(plan, n, p0):
    """Largest difference of a draw at the rings' points from its whole rings', over the deviation."""
    whole = plan.sample(3, 2).double().cpu().numpy()
    plan.set_rings(n, p0)
    got = plan.sample(3, 2).double().cpu().numpy()
    off, worst = np.concatenate([[0], np.cumsum(n)]), 0.0
    for r in range(2):
        for k in range(len(n)):
            c = np.fft.rfft(whole[r, k]) / plan.n_phi
            phi = p0[k] + 2 * np.pi * np.arange(n[k]) / n[k]
            ref = np.concatenate([_points(c, v) for v in np.array_split(phi, 1 + n[k] // 2048)])
            worst = max(worst, rel_err(got[r, off[k]:off[k + 1]], ref, whole.std()))
    return worst


def test_large_primes_in_fp32():
    """2 x 4079 and 2 x 2039 points: a point is a sum of as many terms; in parts its rounding stays near
    2^-25 sqrt(255) of sums up to three deviations, 1.5e-6 at five times that scatter."""
    from paper_1709_10314_gb300 import Plan
    plan = Plan([30.0], 1.0, 4, 8192, anchor_spacing=2)
    assert _worst(plan, [8158, 4078, 8158, 4078], [0.0, 0.1, 0.2, 0.0]) < 4e-6


@pytest.mark.parametrize("fp64,kappa,n_phi,H", [
    (False, (6.0, 11.0, 25.0), 8192, 2),   # three factors: the largest states
    (False, (6.0, 11.0, 25.0), 8192, 0),
    (True, (6.0, 11.0, 25.0), 4096, 2),
    (True, (6.0, 11.0, 25.0), 4096, 0),
    (True, (9.0,), 8192, 0),               # Alg. 2's order, whose single segment per chain has no right anchor
    (True, (6.0, 15.0), 8192, 0),
    (False, (9.0,), 16384, 0),
    (False, (6.0, 15.0), 8192, 2),
])
def test_longest_rings_of_every_kind_of_plan(fp64, kappa, n_phi, H):
    """Bounds: FP32 sums as above (more for the modes' phases); FP64 phases m phi0 of up to 8192 x 0.3 rad
    round to 2.7e-13."""
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, SMERF_RECUR_FP64, Plan
    flags = (SMERF_RECUR_FP64 if fp64 else 0) | (0 if H else SMERF_ORDER_PAPER)
    plan = Plan(list(kappa), 1.0, 8, n_phi, flags=flags, anchor_spacing=H)
    n = [12, n_phi // 2, n_phi - 2, n_phi, n_phi - 34, n_phi, 502, n_phi // 4]
    assert _worst(plan, n, [0.1, -0.2, 0.3, 0.0, 0.0, 0.25, 0.3, 0.0]) < (1e-11 if fp64 else 1e-5)


def _layout(kind, n_theta, n_phi):
    """whole rings with offsets; the same with short rings of every kind among them (2 x prime, ends on 8
    bytes); or every second ring short (at most n_phi / 2 points)."""
    n, p0 = [n_phi] * n_theta, [0.0 if k % 3 == 0 else 0.07 * k for k in range(n_theta)]
    short = {"whole": [], "few": [1, n_theta - 1], "many": range(0, n_theta, 2)}[kind]
    for i, k in enumerate(short):
        n[k] = min(n_phi // 2, (6, 62, n_phi // 2, 4, n_phi // 4, 2 * 37, n_phi // 2 - 2)[i % 7])
    return n, p0


@pytest.mark.parametrize("p,n_theta,n_phi,H,kind,n", [
    (1, 33, 256, 16, "few", 399),     # four realisations per CTA, a ragged last group
    (2, 17, 512, 4, "few", 121),
    (2, 17, 512, 4, "whole", 121),
    (1, 17, 1024, 4, "few", 140),
    (3, 17, 1024, 4, "few", 130),
    (3, 17, 256, 4, "few", 70),
    (2, 18, 2048, 4, "many", 203),
    (1, 18, 4096, 4, "many", 65),
])
def test_same_draws_on_either_kernel(p, n_theta, n_phi, H, kind, n):
    """Many draws at once on the warp-specialised kernel, one by one on the band kernel: the same bits (the same
    operations in the same order)."""
    import torch
    from graph_util import captured
    from paper_1709_10314_gb300 import SMERF_TABLES_FP32, SMERF_TABLES_FP64, Plan
    for tables in (SMERF_TABLES_FP32, SMERF_TABLES_FP64):
        plan = Plan([6.0, 15.0, 40.0][:p], 1.0, n_theta, n_phi, flags=tables, anchor_spacing=H)
        plan.set_rings(*_layout(kind, n_theta, n_phi))
        got, one = plan.sample(11, n), plan.sample(11, 1)
        for out, kernel in ((got, "segment_ws_kernel"), (one, "segment_band_kernel")):
            assert kernel in captured(lambda: plan.sample(11, len(out), out=out))[0][-1]
        got = plan.sample(11, n)
        for r in (0, 1, 2, 3, n // 2, n - 2, n - 1):
            assert torch.equal(got[r], plan.sample(11 + r, 1)[0])


@pytest.mark.parametrize("kind", ["whole", "few", "many"])
@pytest.mark.parametrize("p,n_phi,H", [(1, 2048, 4), (2, 2048, 4), (3, 2048, 4), (2, 4096, 4), (1, 8192, 4), (2, 8192, 4),
                                        (3, 8192, 4), (1, 16384, 0), (2, 4096, 0)])
def test_long_rings_on_the_warp_specialised_kernel(p, n_phi, H, kind):
    """Bounds as above: FP32 phases and sums."""
    from graph_util import captured
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, Plan
    import torch
    plan = Plan([6.0, 15.0, 40.0][:p], 1.0, 9, n_phi, flags=0 if H else SMERF_ORDER_PAPER, anchor_spacing=H)
    n, p0 = _layout(kind, 9, n_phi)
    assert _worst(plan, n, p0) < 1e-5
    if kind == "whole" and n_phi > 2048:
        out = torch.empty(2, plan.points, device="cuda")
        assert "segment_ws_kernel" in captured(lambda: plan.sample(3, 2, out=out))[0][-1]
