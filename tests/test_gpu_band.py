"""The band kernel and the anchor tiles (small requests, ring-dependent longitudes) against the
warp-specialised kernels that a batch runs the same requests on (the same field bit for bit: the
same operations in the same order), and rings of their own point counts against the oracle."""
import math

import numpy as np
import pytest

import oracle
from gpu_util import oracle_std, rel_err

pytestmark = pytest.mark.gpu
KAPPA = {1: (9.0,), 2: (6.0, 15.0), 3: (6.0, 11.0, 25.0)}


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("p,n_theta,n_phi,H,n", [
    (1, 2, 8, 0, 1),          # the smallest grid: two units
    (1, 9, 16, 2, 3),         # anchor tiles with idle lanes, segments of two rings
    (1, 33, 64, 3, 5),        # odd ring count, ragged last segments, more CTAs than SMs
    (2, 32, 64, 0, 301),      # Alg. 2's order; many realisations
    (2, 40, 128, 4, 2),
    (2, 21, 512, 16, 1),      # fewer than four anchors: no tiles
    (1, 130, 256, 8, 1),      # a chain of more anchors than a tile's chunk
    (2, 70, 1024, 5, 2),      # chunks shorter than a segment
    (3, 40, 64, 4, 3),
    (3, 27, 256, 5, 1),
    (1, 34, 2048, 16, 40),    # FP32: the longest ring the band kernel takes
    (2, 33, 64, 5, 401),      # FP64: two realisations per CTA, an odd count of them, chunks that end mid-segment
    (1, 20, 32, 0, 1025),
    (3, 24, 64, 6, 257),
    (1, 36, 1024, 16, 30),    # FP64, p = 1: many CTAs of 512 threads
    (1, 20, 2048, 0, 3),      # the longest rings, few CTAs: one ring per chunk and a segment in many parts
    (2, 33, 2048, 16, 2),
])
def test_same_field_as_the_batch_kernels(fp64, p, n_theta, n_phi, H, n):
    import torch
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, SMERF_RECUR_FP64, SMERF_TABLES_FP64, Plan, sample_batched
    for flags in (SMERF_RECUR_FP64,) if fp64 else (0, SMERF_TABLES_FP64):
        plan = Plan(list(KAPPA[p]), 1.0, n_theta, n_phi, flags=flags | (0 if H else SMERF_ORDER_PAPER), anchor_spacing=H)
        got = plan.sample(11, n)
        ref = torch.full_like(got, float("nan"))
        sample_batched([plan], [11], [n], [ref])
        assert torch.equal(got, ref)
        # a request's realisations do not depend on how many are drawn with them
        assert torch.equal(plan.sample(11 + n - 1, 1)[0], got[n - 1])


# point counts of every kind (powers of two, 2 x prime, odd halves, whole rings behind rings that
# end on 8 bytes), offsets of either sign and beyond a turn
RINGS = [4, 6, 10, 64, 22, 34, 64, 12, 62, 64, 8, 16, 58, 30, 64]
OFFSETS = [0.3, -0.2, 1e-9, 0.05, 7.5, -9.0, 0.0, math.pi, 2.1, -1e-4, 0.0, 0.7, math.pi / 2, 0.0, 2 * math.pi]


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("p,H", [(1, 4), (2, 0), (3, 3)])
def test_rings_of_their_own_point_counts(fp64, p, H):
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, SMERF_RECUR_FP64, Plan
    flags = (SMERF_RECUR_FP64 if fp64 else 0) | (0 if H else SMERF_ORDER_PAPER)
    plan = Plan(list(KAPPA[p]), 1.0, len(RINGS), 64, flags=flags, anchor_spacing=H)
    plan.set_rings(RINGS, OFFSETS)
    got = plan.sample(5, 2).cpu().numpy()
    ref = oracle.sample_rings(list(KAPPA[p]), 1.0, len(RINGS), RINGS, OFFSETS, 5, n_samples=2, H=H, n_phi=64)
    ref = np.stack([np.concatenate(r) for r in ref])
    assert rel_err(got, ref, oracle_std(KAPPA[p], 1.0, len(RINGS), 64)) < (1e-10 if fp64 else 1e-4)


def test_long_rings_of_their_own_point_counts():
    """Rings on thread groups of 64 threads up to the whole CTA, with large prime factors: against
    the same plan's whole rings, whose spectrum the few points sample (FP64, no aliasing: the point
    counts carry every mode that is above rounding)."""
    import torch
    from paper_1709_10314_gb300 import SMERF_RECUR_FP64, Plan
    for n_phi, n in ((1024, 998), (2048, 2026), (4096, 4058)):  # 2 x 499, 2 x 1013, 2 x 2029
        plan = Plan([5.0], 1.0, 6, n_phi, flags=SMERF_RECUR_FP64)
        whole = plan.sample(3, 1)[0].cpu().numpy()
        plan.set_rings([n] * 6, [0.1] * 6)
        got = plan.sample(3, 1)[0].cpu().numpy().reshape(6, n)
        torch.cuda.synchronize()
        for k in range(6):
            c = np.fft.rfft(whole[k]) / n_phi
            assert rel_err(got[k], oracle.ring_values(np.concatenate([c[:-1], [c[-1].real]]), n, 0.1), whole.std()) < 1e-11  # phases of up to 1.3e4 rad in FP64
