"""The staged streaming passes at the edges of their dispatch: less than a group, a range and its
neighbours, the last size whose ranges are staged whole and the first that is not, and the size from
which four ranges share a block (FP16 and FP32), with image pairs that end inside a group.

Checks per size: the loss against the FP64 sum over the exported residuals and weights (the residual
export is another kernel), and the gradient against the quadratic form's at the same poses (another
accumulation). Both sides hold FP32 sums of at most 2,048 terms of one range, added up with
compensation, so they agree to 2048^0.5 x 2^-24 = 3e-6 of the sum of magnitudes: 1e-5 of the loss (all
its terms are positive) and 1e-4 of the largest gradient component (whose terms cancel by less
than a factor of ten here, with an outlier-like scene). The fused reweighting pass must give
the kept count and weights of the separate one, bit for bit."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu

WR = 2048
SIZES = [3, 33, WR - 1, WR, WR + 1, 3 * WR + 65, 304 * WR, 304 * WR + 1, 45600 * WR - 5, 45600 * WR - WR - 5]


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("n", SIZES)
def test_pass_covers_every_point_pair_once(n, storage):
    build.build()
    rng = np.random.default_rng(n % 1000)
    ang = np.arange(4) * np.pi / 8
    R = np.stack([O.expmap(np.array([0.0, a, 0.0]) + 0.02 * rng.normal(size=3)) for a in ang])
    c = np.stack([3 * np.sin(ang), 0.1 * rng.normal(size=4), -3 * np.cos(ang)], 1)
    t = -np.einsum("nab,nb->na", R, c)
    ci, cj = np.array([0, 1, 0], np.int32), np.array([1, 2, 3], np.int32)
    cuts = [0, max(1, n // 3), max(2, 2 * n // 3 - 1), n]
    pid = torch.repeat_interleave(torch.arange(3, dtype=torch.int32, device="cuda"),
                                  torch.tensor(np.diff(cuts), device="cuda"))
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x1, x2 = (torch.rand(n, 2, generator=g, device="cuda") - 0.5 for _ in range(2))
    opt = fm.default_options(storage=storage, delta=1e-3)
    with fm.Problem(R, t, ci, cj, pid, x1, x2, options=opt) as p:
        kept = p.irls_weights(0.2)
        w = p.get_weights()
        e = p.residuals()
        loss, grad = p.loss_grad()
        ref = float(np.sum(w.astype(np.float64) * e.astype(np.float64) ** 2)) / n
        assert loss == pytest.approx(ref, rel=1e-5)
        p.preaggregate()
        lq, gq = p.loss_grad_quadratic()
        assert np.abs(grad - gq).max() <= 1e-4 * np.abs(grad).max()
        assert p.step_irls(0.2, 1, count=True) == kept == int((w > 0).sum())
        assert np.array_equal(p.get_weights(), w)
    with fm.Problem(R, t, ci, cj, pid, x1, x2, options=fm.default_options(storage=storage, loss="l1")) as p:
        assert p.loss_grad()[0] == pytest.approx(float(np.abs(e.astype(np.float64)).mean()), rel=1e-5)
