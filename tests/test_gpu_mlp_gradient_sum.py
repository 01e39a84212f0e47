"""The network's gradient without a step is the one the step takes: its sums over the blocks' partials on the
device, for one block, two, the most blocks and several tiles a block. Linear in the samples: the gradient of a batch is the mean of
the gradients of its halves within FP32 rounding (sums of at most 304 partials of sums of 64 terms: 2^-24 x 368 =
2.2e-5 of the sum of magnitudes; terms of one sign within a factor of 20, so 5e-4 of the largest component).
A call must not cost several steps: it did when the host added the partials up (8.6 steps at 16,384 samples,
1.1 with the sums on the device; 4 are allowed)."""
import time

import numpy as np
import pytest
import torch

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build, learned

pytestmark = pytest.mark.gpu


def _batch(n):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    return (torch.randn(n, 8, generator=g, device="cuda").to(torch.bfloat16),
            (torch.rand(n, generator=g, device="cuda") < 0.5).float())


@pytest.mark.parametrize("n", [2, 128, 16384, 64 * 304 * 2, 65536])
def test_gradient_is_the_mean_of_its_halves(n):
    build.build()
    net = fm.Mlp(learned.init_params(1))
    x, y = _batch(n)
    loss, g = net.gradient(x, y)
    la, ga = net.gradient(x[: n // 2], y[: n // 2])
    lb, gb = net.gradient(x[n // 2:].contiguous(), y[n // 2:].contiguous())
    assert loss == pytest.approx((la + lb) / 2, rel=1e-5)
    assert np.abs(g - (ga + gb) / 2).max() <= 5e-4 * np.abs(g).max()
    assert np.array_equal(net.gradient(x, y)[1], g)


def test_gradient_costs_no_more_than_a_few_steps():
    build.build()
    net = fm.Mlp(learned.init_params(1))
    x, y = _batch(16384)

    def seconds(f):
        out = []
        for _ in range(40):
            t = time.perf_counter()
            f()
            out.append(time.perf_counter() - t)
        return np.median(out)
    step = seconds(lambda: net.train_step(x, y, 0.0))
    assert seconds(lambda: net.gradient(x, y)) <= 4 * step
