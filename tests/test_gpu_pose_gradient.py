"""The backward kernel of the torch objective against the torch operations it replaces, at the edges
of its blocks, and the calls that must still take those operations: a backward that is itself
differentiated, float32 and non-contiguous rotations. Both are two FP64 products and one sum per entry:
they agree to 4 roundings, 1e-15 of the largest entry."""
import numpy as np
import pytest
import torch

import scenegen
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import autograd, binding, build

pytestmark = pytest.mark.gpu


def _torch_ops(grad, R, scale):
    g = grad * scale
    return 0.5 * autograd._hat(g[:, :3]) @ R, g[:, 3:]


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1000])
def test_kernel_equals_torch_operations(n):
    build.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    grad = torch.randn(n, 6, dtype=torch.float64, device="cuda", generator=g)
    R = torch.randn(n, 3, 3, dtype=torch.float64, device="cuda", generator=g)
    s = torch.tensor(-1.7, dtype=torch.float64, device="cuda")
    for a, b in zip(binding.pose_gradient(grad, R, s), _torch_ops(grad, R, s)):
        assert a.shape == b.shape and (a - b).abs().max() <= 1e-15 * b.abs().max()


def test_other_inputs_take_the_torch_operations():
    sc = scenegen.make_scene("ring16", seed=3)
    R0 = sc.R_init.cuda()
    C0 = (-(sc.R_init.transpose(1, 2) @ sc.t_init[:, :, None])[:, :, 0]).cuda()
    with fm.Problem(sc.R_init, sc.t_init, sc.cam_i, sc.cam_j, sc.pair_id, sc.x1, sc.x2) as p:
        def grads(R, C, **kw):
            return torch.autograd.grad(2.0 * fm.epipolar_loss(p, R, C), (R, C), **kw)

        R, C = R0.clone().requires_grad_(), C0.clone().requires_grad_()
        ref = grads(R, C)
        again = grads(R, C, create_graph=True)
        for a, b in zip(ref, again):
            assert (a - b).abs().max() <= 1e-15 * b.abs().max()
        # the backward's own graph: the gradient is linear in R
        torch.autograd.grad(again[0].sum(), R)
        Rt = R0.transpose(1, 2).contiguous().transpose(1, 2).requires_grad_()
        assert not Rt.is_contiguous()
        for a, b in zip(ref, grads(Rt, C)):
            assert (a - b).abs().max() <= 1e-15 * b.abs().max()
        R32 = R0.float().requires_grad_()
        g32 = grads(R32, C)
        assert g32[0].dtype == torch.float32 and (g32[0] - ref[0]).abs().max() <= 1e-3 * ref[0].abs().max()
        loss = torch.empty(1, dtype=torch.float64, device="cuda")
        grad = torch.empty(sc.n_cams, 6, dtype=torch.float64, device="cuda")
        p.loss_grad_device(loss, None)
        p.loss_grad_device(None, grad)
        l, g = p.loss_grad()
        assert loss.item() == l == p.last_loss() and np.array_equal(grad.cpu().numpy(), g)
