"""A refused allocation: reported once, and forgotten.  The allocations are larger than what the
device has left, so they are refused before any memory is touched."""
import numpy as np
import pytest

from paper_1202_6351_gb300 import lbm, workloads

pytestmark = pytest.mark.gpu

OMEGAS = (1.1, 1.7, 1.7, 1.0, 1.2, 0.9)
HUGE = (32768, 65535)  # 155 GB in FP64


def test_a_refused_allocation_is_not_reported_by_later_calls():
    import torch

    torch.cuda.init()
    fields = workloads.random_fields(3, 40, 30, u_amp=0.03, rho_amp=0.01)
    with lbm.Lattice(40, 30, OMEGAS) as L, lbm.Lattice(40, 30, OMEGAS) as ref:
        ref.init(*fields).step(20)
        held = []
        try:
            with pytest.raises(lbm.LBMError) as e:
                for _ in range(4):
                    held.append(lbm.Lattice(*HUGE, OMEGAS, store=lbm.F64))
            assert e.value.code == lbm.LBM_ENOMEM
            L.init(*fields).step(20)
            np.testing.assert_array_equal(L.get_f(), ref.get_f())
            assert float(torch.ones(8, device="cuda").sum()) == 8.0
        finally:
            for h in held:
                h.close()


def test_memory_that_pytorch_holds_unused_is_given_back():
    """PyTorch's caching allocator keeps freed tensors; a lattice that needs their memory gets it."""
    import torch

    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    block = torch.empty(int(total * 0.55), dtype=torch.uint8, device="cuda")
    del block
    assert torch.cuda.memory_reserved() > 0.5 * total
    try:
        with lbm.Lattice(*HUGE, OMEGAS, store=lbm.F64) as L:
            assert L.time == 0
    finally:
        torch.cuda.empty_cache()
