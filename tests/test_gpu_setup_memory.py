"""Device memory that plan creation leaves in the library's scratch pool."""
import pytest

pytestmark = pytest.mark.gpu


def _kept(make):
    """Bytes that smerf_scratch_trim returns after make()."""
    import torch
    from paper_1709_10314_gb300 import scratch_trim
    torch.cuda.synchronize()
    scratch_trim()
    plans = make()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    scratch_trim()
    kept = torch.cuda.mem_get_info()[0] - free
    for p in plans:
        p.close()
    return kept


def test_overlapped_set_ups_keep_a_bounded_part_of_the_pool():
    """16 set-ups of 2 x 67 MB of temporaries at once: three fit the 512 MB that set-ups may keep (the pool maps
    32 MB at a time), not 2.1 GB; a single set-up keeps its own."""
    from paper_1709_10314_gb300 import Plan, create_plans
    spec = dict(kappa=[20.0, 50.0], A=1.0, n_theta=2048, n_phi=4096)
    assert _kept(lambda: create_plans([dict(spec) for _ in range(16)])) < 640 << 20
    assert 134 << 20 <= _kept(lambda: [Plan([20.0, 50.0], 1.0, 2048, 4096)]) < 256 << 20
    # the share is given back: the next ones pool again
    assert _kept(lambda: create_plans([dict(spec)])) >= 134 << 20
