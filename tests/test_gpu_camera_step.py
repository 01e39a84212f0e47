"""The camera step at the edges of its dispatch: one camera a block and four warps (up to 1,216 cameras with
more than 44 items each), two cameras of two warps (up to 2,432), eight of one warp beyond; cameras with more than 32 image pairs, and with more items than the warps take in one pass.

The gradient is compared with the quadratic form's at the same poses, which another kernel sums up per
pair before its chain rule: both hold FP32 sums whose errors are a few 1e-6 of the sum of magnitudes, so
1e-4 of the largest component where the terms cancel by less than a factor of ten. Three steps (with
the geometry records of each new pose written by the step) must give the bits of three evaluations
(which build the records anew) with apply_gradient."""
import numpy as np
import pytest
import torch

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


# cameras, image pairs from a camera to its next ones, point pairs of a pair
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("cams,near,points", [
    (2, 1, 3), (3, 2, 5000), (12, 5, 60000), (70, 34, 40), (152, 3, 31), (153, 3, 33), (160, 4, 20000),
    (200, 40, 700), (1216, 2, 40), (1217, 2, 40), (2432, 1, 9), (2433, 1, 9), (2600, 18, 3)])
def test_step_and_gradient(cams, near, points, storage):
    build.build()
    g = torch.Generator(device="cuda")
    g.manual_seed(cams)
    rng = np.random.default_rng(cams)
    a = 2 * np.pi * np.arange(cams) / max(cams, 8)
    R = np.stack([np.array([[np.cos(x), 0, -np.sin(x)], [0, 1, 0], [np.sin(x), 0, np.cos(x)]]) for x in a])
    c = np.stack([np.sin(a), 0.3 * rng.normal(size=cams), -np.cos(a)], 1) * 4
    t = -np.einsum("nab,nb->na", R, c)
    i = np.repeat(np.arange(cams), near)
    j = i + np.tile(np.arange(1, near + 1), cams)
    keep = j < cams
    i, j = i[keep].astype(np.int32), j[keep].astype(np.int32)
    n = len(i) * points
    pid = torch.arange(len(i), dtype=torch.int32, device="cuda").repeat_interleave(points)
    x1, x2 = (torch.rand(n, 2, generator=g, device="cuda") - 0.5 for _ in range(2))
    opt = fm.default_options(storage=storage, delta=1e-3)
    with fm.Problem(R, t, i, j, pid, x1, x2, options=opt) as p, fm.Problem(R, t, i, j, pid, x1, x2, options=opt) as q:
        for s in (p, q):
            s.irls_weights(0.3)
        grad = p.loss_grad()[1]
        p.preaggregate()
        form = p.loss_grad_quadratic()[1]
        assert np.abs(grad - form).max() <= 1e-4 * np.abs(grad).max()
        p.step(3)
        for _ in range(3):
            q.apply_gradient(q.loss_grad()[1])
        for u, v in zip(p.get_params(), q.get_params()):
            np.testing.assert_array_equal(u, v)
        assert p.loss_grad()[0] == q.loss_grad()[0]


def test_coincident_cameras_are_reported():
    # the pass forms the pair geometry itself, in every iteration of a chain
    build.build()
    rng = np.random.default_rng(0)
    R, t = np.stack([np.eye(3)] * 3), np.array([[0.0, 0, 0], [0, 0, 0], [1, 0, 0]])
    x1, x2 = (rng.uniform(-0.5, 0.5, (40, 2)).astype(np.float32) for _ in range(2))
    pid = np.repeat(np.arange(2, dtype=np.int32), 20)
    for call in (lambda p: p.loss_grad(), lambda p: p.irls_weights(0.1), lambda p: (p.step(1), p.last_loss())):
        with fm.Problem(R, t, np.array([0, 0], np.int32), np.array([1, 2], np.int32), pid, x1, x2) as p:
            with pytest.raises(fm.FastMapError):
                call(p)
