"""The density energy N = 1/2 sum_b A_b rho_b psi_b (Eq. 6) as a
torch.autograd.Function.

forward runs the scatter and the spectral solve (fftpl_energy); backward is
the field-gather kernel (fftpl_gather, mode "gather": the q.E of Eq. 7) or
the exact derivative of the binned energy (mode "adjoint"), scaled by the
incoming gradient.  Positions are float32 CUDA tensors of the problem's
movable cells.

On a stream other than the handle's, the handle's work is ordered after what
that stream holds (the positions, the incoming gradient, the memory of the
outputs) and that stream after the handle's work.  On the handle's own stream
neither direction waits for the device: the energy goes straight into the
output tensor and the gather kernel reads the incoming gradient from the
device.  (With a wait and a copy for the energy and two multiplications after
the gather, forward and backward of 500K cells took 380 us of host time for
70 us of kernels.)
"""
from __future__ import annotations

import torch
from torch.autograd import forward_ad

from . import fftpl as F

_MODES = {"gather": 0, "adjoint": 1}


def _other_stream(problem, device):
    """The current stream if the handle is not ordered with it, else None."""
    cur = torch.cuda.current_stream(device).cuda_stream
    return None if cur == getattr(problem, "stream", None) else cur


def _plain_scalar(g):
    """A float64 CUDA scalar with memory of its own (not, say, a batch of
    gradients under vmap, which has no data pointer) that no graph is being
    recorded for (create_graph: the product with it is differentiable) and that
    carries no forward-mode tangent (the product carries it on); its memory
    holds the value itself, not the negative a view may stand for."""
    if torch.is_grad_enabled() and g.requires_grad:
        return False
    if g.dtype != torch.float64 or not g.is_cuda or g.dim() != 0:
        return False
    try:
        if g.data_ptr() == 0:
            return False
    except RuntimeError:
        return False
    return not g.is_neg() and forward_ad.unpack_dual(g).tangent is None


class DensityEnergy(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, y, problem, mode="gather"):
        if mode not in _MODES:
            raise ValueError(f"mode must be one of {sorted(_MODES)}")
        x = x.detach().contiguous()
        y = y.detach().contiguous()
        other = _other_stream(problem, x.device)
        if other is None:
            N = torch.empty((), dtype=torch.float64, device=x.device)
            F.fftpl_energy_device(problem.h, x, y, N)
        else:
            F.fftpl_order_after(problem.h, other)
            N = torch.tensor(F.fftpl_energy(problem.h, x, y), dtype=torch.float64,
                             device=x.device)
        problem._energy_calls = getattr(problem, "_energy_calls", 0) + 1
        ctx.problem = problem
        ctx.mode = mode
        ctx.call = problem._energy_calls
        ctx.save_for_backward(x, y)
        return N

    @staticmethod
    def backward(ctx, grad_out):
        x, y = ctx.saved_tensors
        problem = ctx.problem
        gx = torch.empty_like(x)
        gy = torch.empty_like(y)
        other = _other_stream(problem, x.device)
        if other is not None:
            F.fftpl_order_after(problem.h, other)
        if problem._energy_calls != ctx.call:
            # the handle's maps belong to a later evaluation: recompute them
            F.fftpl_energy(problem.h, x, y, sync=False)
            problem._energy_calls += 1
        if other is None and _plain_scalar(grad_out):
            F.fftpl_gather_scaled(problem.h, x, y, grad_out, gx, gy, _MODES[ctx.mode])
            return gx, gy, None, None
        F.fftpl_gather(problem.h, x, y, gx, gy, _MODES[ctx.mode])
        if other is not None:
            F.fftpl_order_before(problem.h, other)
        s = grad_out.to(torch.float32)
        return gx * s, gy * s, None, None


def density_energy(x, y, problem, mode="gather"):
    """N(x, y) with the hand-written backward (see DensityEnergy)."""
    return DensityEnergy.apply(x, y, problem, mode)
