"""torch.autograd.Function over the epipolar objective (the differentiation form of the path).

EpipolarLoss.apply(problem, R, c) evaluates the problem's objective (IRLS-weighted or L1,
Sec. "Epipolar Adjustment") at rotations R (N,3,3) and camera centres c (N,3), float64 CUDA
tensors. The forward call is one pass of the library's fused loss/adjoint kernels; the only
thing kept for backward is the per-camera gradient (N x 6), never a per-pair or per-point
quantity. With recompute=True the forward keeps nothing and backward runs the pass again.

Gradients: the library returns the left-trivialised gradient g_phi (R <- Exp(phi) R) and
g_c. For R the backward returns the tangent-space Euclidean gradient 0.5 [g_phi]_x R, whose
inner product with any rotation perturbation [dphi]_x R equals g_phi . dphi, so autograd
through any rotation parameterisation (exponential map, 6D, quaternions) is exact. Contiguous
float64 inputs take one kernel for this (fm_pose_gradient; as torch operations it was 13 launches,
one of them a 70 us batched FP64 matrix product); other types and layouts, tensors whose memory does not
hold their values (a batched backward), and a backward that is itself differentiated (create_graph), take
the torch operations.
"""
from __future__ import annotations

import torch

from .binding import pose_gradient


def _hat(v: torch.Tensor) -> torch.Tensor:
    z = torch.zeros_like(v[:, 0])
    return torch.stack([torch.stack([z, -v[:, 2], v[:, 1]], -1),
                        torch.stack([v[:, 2], z, -v[:, 0]], -1),
                        torch.stack([-v[:, 1], v[:, 0], z], -1)], -2)


def _loss_grad(problem, R, c):
    R = R.detach().to(torch.float64).contiguous()
    c = c.detach().to(torch.float64).contiguous()
    problem.set_params_device(R, c)
    loss = torch.empty((), dtype=torch.float64, device=R.device)
    grad = torch.empty(R.shape[0], 6, dtype=torch.float64, device=R.device)
    problem.loss_grad_device(loss, grad)
    return loss, grad


def _in_memory(t: torch.Tensor) -> bool:
    """A plain tensor or parameter whose memory holds its values, so that a kernel can be given its address. Not so for the
    gradients of a batched backward (no storage of their own, though their Python type is torch.Tensor), for
    a lazily negated tensor (autograd's imaginary parts of conjugates: the memory has the other sign) and
    for autograd's zeros without memory."""
    if type(t) not in (torch.Tensor, torch.nn.Parameter) or t.is_neg():
        return False
    try:
        return t.data_ptr() != 0
    except RuntimeError:
        return False


class EpipolarLoss(torch.autograd.Function):
    @staticmethod
    def forward(ctx, problem, R, c, recompute: bool = False):
        loss, grad = _loss_grad(problem, R, c)
        ctx.problem = problem
        ctx.recompute = recompute
        if recompute:
            ctx.save_for_backward(R, c)
        else:
            ctx.save_for_backward(R, grad)
        return loss

    @staticmethod
    def backward(ctx, grad_out):
        if ctx.recompute:
            R, c = ctx.saved_tensors
            _, grad = _loss_grad(ctx.problem, R, c)
        else:
            R, grad = ctx.saved_tensors
        # (saved-tensor hooks may give back other devices, layouts and shapes than were saved)
        if (not torch.is_grad_enabled() and R.dtype == grad.dtype == grad_out.dtype == torch.float64
                and R.is_cuda and grad_out.get_device() == grad.get_device() == R.get_device()
                and R.shape == (grad.shape[0], 3, 3) and grad.shape[1:] == (6,)
                and R.is_contiguous() and grad.is_contiguous()
                and _in_memory(R) and _in_memory(grad) and _in_memory(grad_out)):
            return None, *pose_gradient(grad, R, grad_out), None
        g = grad * grad_out
        gR = 0.5 * _hat(g[:, :3]) @ R.to(torch.float64)
        return None, gR.to(R.dtype), g[:, 3:].to(R.dtype), None


def epipolar_loss(problem, R, c, recompute: bool = False) -> torch.Tensor:
    """Differentiable objective of `problem` (a binding.Problem) at (R, c)."""
    return EpipolarLoss.apply(problem, R, c, recompute)
