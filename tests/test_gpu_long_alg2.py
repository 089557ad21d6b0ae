"""Rings of 8192 complex points without anchors (Alg. 2's order, or fewer rings than an anchor spacing),
which the warp-specialised kernel holds: its tables are the ones it reads, in either precision."""
import pytest

from gpu_util import rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_theta,paper", [(8, True), (8, False), (33, True)])
def test_same_field_with_either_tables(n_theta, paper):
    """FP32 recursion against the FP64 mode on the same noise (bound of the FP32 parity tests), from FP32
    and from FP64 tables; the tables' entries are the same to FP32 rounding."""
    import numpy as np
    import torch
    from paper_1709_10314_gb300 import SMERF_ORDER_PAPER, SMERF_RECUR_FP64, SMERF_TABLES_FP32, SMERF_TABLES_FP64, Plan
    order = SMERF_ORDER_PAPER if paper else 0
    plans = [Plan([30.0], 1.0, n_theta, 16384, flags=order | f)
             for f in (SMERF_RECUR_FP64, SMERF_TABLES_FP32, SMERF_TABLES_FP64)]
    assert plans[1].info()["anchor_spacing"] == 0
    ref, t32, t64 = (p.sample(7, 2).double().cpu().numpy() for p in plans)
    torch.cuda.synchronize()
    assert rel_err(t32, ref, ref.std()) < 1e-4 and rel_err(t64, ref, ref.std()) < 1e-4
    a, b = plans[1].tables(1, 0, 1), plans[2].tables(1, 0, 1)
    assert np.allclose(a, b, rtol=2e-7, atol=1e-30)
