"""The FP64 mode's fixed-point ring FFT on the GPU against rings of half the points, which the mixed-radix
passes synthesise in FP64 from the same coefficients: every second value of a whole ring."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_phi", [8, 64, 512, 2048, 4096])
@pytest.mark.parametrize("kappa,n", [((3000.0,), 3), ((20.0, 50.0), 3), ((3000.0,), 200)])
def test_every_second_point_of_a_whole_ring(kappa, n_phi, n):
    """kappa = 3000: a flat spectrum, the fixed point's hardest.  Bound: seven roundings (fold, packing, five
    passes) of at most 2.2e-16 each on the FP64 side, 6e-16 of the deviation by scatter, less on the
    fixed-point side, and 6.5 times that for the largest of up to 1e6 values."""
    import torch
    from paper_1709_10314_gb300 import SMERF_RECUR_FP64, Plan
    n_theta, theta = 12, None
    if kappa[0] > 1000:  # rings so close that the tables resolve kappa (its steps grow as e^(kappa dtheta))
        theta = [1.5 + 0.01 * k for k in range(n_theta)]
    if n * n_theta * n_phi > 2e6:
        n = 40
    plan = Plan(list(kappa), 1.0, n_theta, n_phi, flags=SMERF_RECUR_FP64, anchor_spacing=4, theta=theta)
    whole = plan.sample(5, n)
    plan.set_rings([n_phi // 2] * n_theta)
    half = plan.sample(5, n).view(n, n_theta, n_phi // 2)
    err = float((whole[:, :, ::2] - half).abs().max() / whole.std())
    assert err < 4e-15


@pytest.mark.parametrize("n_phi,n,H", [(64, 3, 4), (64, 1500, 4), (1024, 2, 4), (1024, 200, 4), (4096, 2, 0)])
def test_rings_with_coefficients_that_are_not_finite(n_phi, n, H):
    """A kappa that 12 rings do not resolve (its step grows as e^785) overflows the tables: the rings whose
    coefficients are not finite are NaN throughout, as FP32's are, and no others."""
    import torch
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, SMERF_RECUR_FP64, SMERF_TABLES_FP32, Plan
    flags = SMERF_TABLES_FP32 | (0 if H else SMERF_ORDER_PAPER)
    f32, f64 = (Plan([3000.0], 1.0, 12, n_phi, flags=flags | f, anchor_spacing=H).sample(5, n) for f in (0, SMERF_RECUR_FP64))
    bad = torch.isnan(f64)
    assert bool(bad.any()) and bool((bad.any(2) == bad.all(2)).all())
    assert torch.equal(bad.any(2), torch.isnan(f32).any(2))
    assert bool(torch.isfinite(f64[~bad]).all())
