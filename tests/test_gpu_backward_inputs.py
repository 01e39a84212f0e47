"""Incoming gradients and saved tensors of the torch objective's backward that its kernel must not be given
as they lie in memory, against the plain backward scaled by hand. Both take FP64 products and one sum per
entry: they agree to 4 roundings, 1e-15 of the largest entry."""
import pytest
import torch

import scenegen
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import autograd, build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scene():
    build.build()
    sc = scenegen.make_scene("ring16", seed=3)
    R = sc.R_init.cuda()
    C = (-(sc.R_init.transpose(1, 2) @ sc.t_init[:, :, None])[:, :, 0]).cuda()
    with fm.Problem(sc.R_init, sc.t_init, sc.cam_i, sc.cam_j, sc.pair_id, sc.x1, sc.x2) as p:
        leaves = R.clone().requires_grad_(), C.clone().requires_grad_()
        yield p, R, C, torch.autograd.grad(fm.epipolar_loss(p, *leaves), leaves)


def _same(got, ref):
    for a, b in zip(got, ref):
        assert a.shape == b.shape and (a - b).abs().max() <= 1e-15 * b.abs().max()


@pytest.mark.parametrize("recompute", [False, True])
def test_batched_backward(scene, recompute):
    p, R, C, ref = scene
    s = torch.tensor([1.0, -2.5, 0.0], dtype=torch.float64, device="cuda")
    leaves = R.clone().requires_grad_(), C.clone().requires_grad_()
    loss = fm.epipolar_loss(p, *leaves, recompute)
    got = torch.autograd.grad(loss, leaves, s, is_grads_batched=True)
    for k in range(3):
        _same([g[k] for g in got], [s[k] * g for g in ref])


def test_lazily_negated_gradient(scene):
    p, R, C, ref = scene
    leaves = R.clone().requires_grad_(), C.clone().requires_grad_()
    two = torch.tensor(2.0, dtype=torch.float64, device="cuda")
    neg = torch._neg_view(two)
    assert neg.is_neg() and neg.item() == -2.0
    _same(torch.autograd.grad(fm.epipolar_loss(p, *leaves), leaves, neg), [-2.0 * g for g in ref])


def test_zero_gradient_without_memory(scene):
    p, R, C, _ = scene
    leaves = R.clone().requires_grad_(), C.clone().requires_grad_()
    zero = torch._efficientzerotensor((), dtype=torch.float64, device="cuda")
    for g in torch.autograd.grad(fm.epipolar_loss(p, *leaves), leaves, zero):
        assert not g.any()


def test_saved_gradient_in_another_layout(scene):
    p, R, C, ref = scene
    leaves = R.clone().requires_grad_(), C.clone().requires_grad_()
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t.transpose(0, 1).contiguous(), lambda t: t.transpose(0, 1)):
        loss = fm.epipolar_loss(p, *leaves)
    _same(torch.autograd.grad(loss, leaves), ref)
    # the gradient alone: R comes back as it was
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t.t().contiguous() if t.dim() == 2 else t,
                                                  lambda t: t.t() if t.dim() == 2 else t):
        loss = fm.epipolar_loss(p, *leaves)
    _same(torch.autograd.grad(loss, leaves), ref)


def test_parameters_take_the_kernel(scene, monkeypatch):
    p, R, C, ref = scene
    calls = []
    kernel = autograd.pose_gradient
    monkeypatch.setattr(autograd, "pose_gradient", lambda *a: calls.append(a) or kernel(*a))
    leaves = torch.nn.Parameter(R.clone()), torch.nn.Parameter(C.clone())
    fm.epipolar_loss(p, *leaves).backward()
    _same([v.grad for v in leaves], ref)
    assert len(calls) == 1 and type(leaves[0].grad) is torch.Tensor
