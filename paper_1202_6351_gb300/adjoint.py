"""Differentiable cascaded run: a torch.autograd.Function over lbm_adjoint_run.

``final_velocity_loss(u0, force, omega_shear, target, nsteps, every)`` returns
L = 1/2 sum |u(T) - target|^2 for a periodic cascaded lattice started at the
transformed equilibrium with velocity u0 (rho = rho0), driven by the per-node
body force ``force`` [2, ny, nx], with shear rate omega_4 = omega_5 =
``omega_shear`` and the other rates fixed.  Its backward pass returns the
gradients the CUDA adjoint computed in the same call (reverse streaming plus
the transposed collision, checkpoints every ``every`` steps, FP64
accumulation).  All tensors are float64 on the current CUDA device.  The states
of a run may stay in PyTorch's caching allocator after the call (KEPT_PART).
"""
from __future__ import annotations

import torch

from . import lbm


# The checkpoints of a run live in PyTorch's caching allocator, on the stream the lattice runs on, if they
# take at most this part of the device memory (18.6 of 298 GB): a training loop maps them once instead of on
# every call (ms per call mapped on each call -> kept: 512^2, 400 steps, 1.0 GB 10.6 -> 8.4; 2048^2, 100 steps,
# 4.0 GB 35.2 -> 27.0, 15.5 GB 58.4 -> 27.3).  PyTorch keeps that memory until torch.cuda.empty_cache(), which
# lbm.py calls when an allocation of the library finds no room.  Larger runs, and runs that find no room in
# the allocator, use memory that the library maps for the call.
KEPT_PART = 1 / 16


def _workspace(nbytes):
    if nbytes > KEPT_PART * torch.cuda.get_device_properties(torch.cuda.current_device()).total_memory:
        return None
    try:
        return torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    except torch.cuda.OutOfMemoryError:
        return None


class FinalVelocityLoss(torch.autograd.Function):
    @staticmethod
    def forward(ctx, u0, force, omega_shear, target, nsteps, every, other_rates, store):
        ny, nx = u0.shape[1], u0.shape[2]
        w = float(omega_shear)
        rates = (other_rates[0], w, w, other_rates[1], other_rates[2], other_rates[3])
        stream = torch.cuda.current_stream().cuda_stream
        with lbm.Lattice(nx, ny, rates, model=lbm.CASCADED, store=store, stream=stream) as L:
            L.set_force_field(force.detach().contiguous())
            ws = _workspace(L.adjoint_workspace(nsteps, every))
            loss, gu, gf, gom = L.adjoint_run(nsteps, every, u0.detach().contiguous(), target.detach().contiguous(),
                                              workspace=ws)
        ctx.save_for_backward(gu, gf)
        # tied shear rate: omega_4 and omega_5 both follow omega_shear
        ctx.g_omega = float(gom[1] + gom[2])
        return torch.tensor(loss, dtype=torch.float64, device=u0.device)

    @staticmethod
    def backward(ctx, g):
        gu, gf = ctx.saved_tensors
        g_omega = torch.tensor(ctx.g_omega, dtype=torch.float64, device=g.device)
        return g * gu, g * gf, g * g_omega, None, None, None, None, None


def final_velocity_loss(u0, force, omega_shear, target, nsteps, every=100, other_rates=(1.0, 1.0, 1.0, 1.0),
                        store=lbm.F32):
    """other_rates = (omega_3, omega_6, omega_7, omega_8)."""
    if not torch.is_tensor(omega_shear):
        omega_shear = torch.tensor(float(omega_shear), dtype=torch.float64, device=u0.device)
    return FinalVelocityLoss.apply(u0, force, omega_shear, target, int(nsteps), int(every), tuple(other_rates),
                                   int(store))
