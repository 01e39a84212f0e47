"""The streaming passes where a range of 2,048 point pairs holds many image pairs: they form the pairs' matrices 16
at a time, so 15, 16, 17, 32 and 33 image pairs in the first range, whose last one ends with the range or behind
it, and the same again in the ranges that follow. One image pair more or less in a table would put a
wrong matrix to a whole image pair.

Checks: the fused reweighting pass gives the count and weights of the separate one (whose matrices come from
geometry records), bit for bit; the loss is the FP64 sum over the exported residuals and weights; the gradient is
that of the evaluation without allocation (records, one thread per image pair) and of the quadratic form. Sums of at most 2,048
FP32 terms on either side: 2048^0.5 x 2^-24 = 3e-6 of the sum of magnitudes, so 1e-5 of the loss (positive
terms) and 1e-4 of the largest gradient component (terms that cancel by less than a factor of ten)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import binding, build

pytestmark = pytest.mark.gpu

WR = 2048


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("over", [0, 37])
@pytest.mark.parametrize("pairs", [15, 16, 17, 32, 33])
def test_many_image_pairs_in_a_range(pairs, over, storage):
    build.build()
    rng = np.random.default_rng(pairs + over)
    first = np.full(pairs, WR // pairs)
    first[: WR - first.sum()] += 1           # ends exactly with the range
    first[-1] += over
    counts = np.concatenate([first, first, first])
    n_pairs, n = len(counts), int(counts.sum())
    n_cams = n_pairs + 1
    ang = 2 * np.pi * np.arange(n_cams) / n_cams
    R = np.stack([O.expmap(np.array([0.0, a, 0.0]) + 0.02 * rng.normal(size=3)) for a in ang])
    c = np.stack([3 * np.sin(ang), 0.1 * rng.normal(size=n_cams), -3 * np.cos(ang)], 1)
    t = -np.einsum("nab,nb->na", R, c)
    ci = np.arange(n_pairs, dtype=np.int32)
    pid = np.repeat(ci, counts)
    x1, x2 = (rng.uniform(-0.5, 0.5, (n, 2)).astype(np.float32) for _ in range(2))
    opt = fm.default_options(storage=storage, delta=1e-3)
    with fm.Problem(R, t, ci, ci + 1, pid, x1, x2, options=opt) as p:
        kept = p.irls_weights(0.2)
        w, e = p.get_weights(), p.residuals()
        assert 0 < kept == int((w > 0).sum()) < n
        loss, grad = p.loss_grad()
        assert loss == pytest.approx(float(np.sum(w.astype(np.float64) * e.astype(np.float64) ** 2)) / n, rel=1e-5)
        p.preaggregate()
        assert np.abs(grad - p.loss_grad_quadratic()[1]).max() <= 1e-4 * np.abs(grad).max()
        if storage == "fp32":
            dev = [torch.as_tensor(a, device="cuda").contiguous() for a in
                   (R, c, ci, ci + 1, np.concatenate([[0], np.cumsum(counts)]).astype(np.int32),
                    np.concatenate([x1, x2], 1), w)]
            lo = torch.zeros(1, dtype=torch.float64, device="cuda")
            go = torch.zeros(n_cams, 6, dtype=torch.float64, device="cuda")
            lib = binding.load_library()
            binding._check(lib.fm_loss_grad_noalloc(n_cams, dev[0].data_ptr(), dev[1].data_ptr(), n_pairs, dev[2].data_ptr(),
                                                    dev[3].data_ptr(), dev[4].data_ptr(), n, dev[5].data_ptr(),
                                                    dev[6].data_ptr(), 0, lo.data_ptr(), go.data_ptr(),
                                                    binding._current_stream()))
            assert lo.item() == pytest.approx(loss, rel=1e-5)
            assert np.abs(grad - go.cpu().numpy()).max() <= 1e-4 * np.abs(grad).max()
        assert p.step_irls(0.2, 1, count=True) == kept
        assert np.array_equal(p.get_weights(), w)
