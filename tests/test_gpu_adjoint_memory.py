"""Device memory of the adjoint: what a run allocates, and what the autograd function keeps in
PyTorch's caching allocator."""
import ctypes as C

import pytest

from paper_1202_6351_gb300 import adjoint, lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps,every", [(16, 4), (200, 200)], ids=["small", "large"])
def test_what_stays_cached_after_a_gradient_is_bounded(steps, every):
    """2048^2 FP32: 151 MB per state, about 1 GB of states and 30 GB; what PyTorch's allocator holds
    afterwards stays below 1/16 of the device memory plus the function's own tensors (six
    fields of 67 MB and their copies)."""
    import torch

    torch.cuda.empty_cache()
    before = torch.cuda.memory_reserved()
    n = 2048
    u0 = torch.zeros((2, n, n), dtype=torch.float64, device="cuda", requires_grad=True)
    force = torch.full((2, n, n), 1e-6, dtype=torch.float64, device="cuda", requires_grad=True)
    omega = torch.tensor(1.6, dtype=torch.float64, device="cuda", requires_grad=True)
    loss = adjoint.final_velocity_loss(u0, force, omega, torch.full_like(u0.detach(), 1e-3), steps, every, store=lbm.F32)
    grads = torch.autograd.grad(loss, (u0, force, omega))
    assert all(bool(torch.isfinite(g).all()) for g in grads)
    limit = torch.cuda.get_device_properties(0).total_memory // 16
    assert torch.cuda.memory_reserved() - before <= limit + 10 * u0.nbytes
    del u0, force, omega, loss, grads
    torch.cuda.empty_cache()


def test_no_force_gradient_array_beside_the_callers():
    """lbm_adjoint_run allocates a force gradient of its own only if the caller takes none."""
    import torch

    torch.cuda.init()
    cudart = C.CDLL("libcudart.so.13")  # the runtime the library is linked with
    used_high = 8  # cudaMemPoolAttrUsedMemHigh
    pool, value = C.c_void_p(), C.c_uint64()
    assert cudart.cudaDeviceGetDefaultMemPool(C.byref(pool), 0) == 0
    u, t, f = (torch.full((2, 512, 512), v, dtype=torch.float64, device="cuda") for v in (0.0, 1e-3, 1e-6))
    high = []
    for want in (True, False):
        with lbm.Lattice(512, 512, (1.1, 1.7, 1.7, 1.0, 1.2, 0.9), store=lbm.F32) as L:
            L.set_force_field(f)
            assert cudart.cudaMemPoolSetAttribute(pool, used_high, C.byref(C.c_uint64(0))) == 0
            L.adjoint_run(4, 2, u, t, want_force=want)
            assert cudart.cudaMemPoolGetAttribute(pool, used_high, C.byref(value)) == 0
            high.append(value.value)
    assert high[1] - high[0] == 2 * 512 * 512 * 8
