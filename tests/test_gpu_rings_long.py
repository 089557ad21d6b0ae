"""Ring-dependent longitudes on long rings, against the same plan's whole rings: their coefficients
evaluated at the rings' own points in FP64."""
import numpy as np
import pytest

from gpu_util import rel_err

pytestmark = pytest.mark.gpu


def _points(c, phi):
    """oracle.ring_values at given longitudes, the Nyquist coefficient's real part at any of them."""
    M = len(c) - 1
    v = c[0].real + 2.0 * (np.exp(1j * np.outer(phi, np.arange(1, M))) @ c[1:M]).real
    return v + c[M].real * np.cos(M * phi)


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
            ref = np.concatenate([_points(c, v) for v in np.array_split(phi, 1 + n[k] // 512)])
            worst = max(worst, rel_err(got[r, off[k]:off[k + 1]], ref, whole.std()))
    return worst


def test_large_primes_in_fp32():
    """2 x 4079 and 2 x 2039 points: a point is a sum of as many terms; in parts of 16 its rounding stays
    near 2^-25 sqrt(255) of sums up to three deviations, 1.5e-6 at five times that scatter."""
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
