"""The network's training step at the edges of its sample tiles: one sample, a tile and its
neighbours, one tile more than the blocks of a launch, the largest batch, and features that are
not 16-byte aligned, against the oracle's gradient and its Adam step.

Tolerance: as for the gradient at ordinary sizes (2e-3 of the largest component): FP32 sums in
another order stay below 1e-5 of it, the rest admits a hidden activation on the other side of a
BF16 rounding boundary. The Adam step of a parameter is lr times a number of magnitude <= 1, and at
the first step that number is the gradient's sign up to eps, so parameters whose gradient exceeds
the tolerance move by lr within 1%."""
import numpy as np
import pytest
import torch

from oracle import learned as L
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build, learned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,offset", [(1, 0), (63, 0), (64, 3), (65, 0), (64 * 304 + 1, 8), (65536, 0)])
def test_gradient_and_step_at_tile_edges(n, offset):
    build.build()
    rng = np.random.default_rng(n)
    X = L.bf16_round(rng.normal(0, 2, (n, 8)))
    y = (rng.random(n) < 0.6).astype(np.float32)
    pv = learned.init_params(5)
    store = torch.zeros(n * 8 + offset, dtype=torch.bfloat16, device="cuda")
    store[offset:] = torch.tensor(X, dtype=torch.float32, device="cuda").to(torch.bfloat16).reshape(-1)
    Xd, Yd = store[offset:].view(n, 8), torch.tensor(y, device="cuda")
    net = fm.Mlp(pv)
    loss, g = net.gradient(Xd, Yd)
    l_or, g_or = L.bce_loss_grad_bf16(L.unflatten(pv.astype(np.float64)), X, y.astype(np.float64))
    g_or = L.flatten(g_or)
    tol = 2e-3 * np.abs(g_or).max()
    assert loss == pytest.approx(l_or, rel=1e-3)
    assert np.abs(g - g_or).max() <= tol
    lr = 1e-2
    step_loss = net.train_step(Xd, Yd, lr)
    assert step_loss == pytest.approx(loss, rel=1e-6)
    moved = (net.params().astype(np.float64) - pv) / lr
    sure = np.abs(g_or) > 2 * tol
    assert np.abs(moved[sure] + np.sign(g_or[sure])).max() <= 1e-2
    again = fm.Mlp(pv)
    again.train_step(Xd, Yd, lr)
    assert np.array_equal(again.params(), net.params())
