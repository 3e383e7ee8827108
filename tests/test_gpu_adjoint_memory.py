"""Device memory that the autograd function keeps in PyTorch's caching allocator."""
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
