"""The learned reweighting at the edges of its steps of 64 point pairs: fewer than a step, a step and
its neighbours, a range and its neighbours, and image pairs that end at every position of a step,
for both storages. The fused pass must give the weights, the kept count and (after one iteration) the poses
of the separate passes bit for bit, and every weight must lie within the bound that the element-wise
test derives: against p / max(|e|, delta) with p from the features that the collection kernel
exports (another kernel), through the library's FP32 forward pass, which differs from the tensor cores
by summation order and by hidden activations on the other side of a BF16 boundary (5e-3 of p, as in
the forward test), by the FP16 rounding of a stored weight (2^-11) and by the fast quotient (2^-22)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build, learned

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("n", [3, 63, 64, 65, 2047, 2048, 2049, 3 * 2048 + 97])
def test_steps_and_ranges(n, storage):
    build.build()
    rng = np.random.default_rng(n)
    m = min(20, n)
    ang = np.arange(6) * np.pi / 12
    R = np.stack([O.expmap(np.array([0.0, a, 0.0]) + 0.02 * rng.normal(size=3)) for a in ang])
    c = np.stack([3 * np.sin(ang), 0.1 * rng.normal(size=6), -3 * np.cos(ang)], 1)
    t = -np.einsum("nab,nb->na", R, c)
    ij = [(i, j) for i in range(6) for j in range(i + 1, 6)] * 2
    ci, cj = (np.array(v, np.int32) for v in zip(*ij[:m]))
    cuts = np.sort(rng.choice(np.arange(1, n), m - 1, replace=False))
    pid = np.repeat(np.arange(m, dtype=np.int32), np.diff([0, *cuts, n]))
    x1, x2 = ((rng.random((n, 2)) - 0.5).astype(np.float32) for _ in range(2))
    score = rng.random(n).astype(np.float32)
    net = fm.Mlp(learned.init_params(7))
    opt = fm.default_options(storage=storage, delta=1e-3, lr_rot=1e-3, lr_c=1e-3)
    tau, cap = 0.1, 0.3
    with fm.Problem(R, t, ci, cj, pid, x1, x2, options=opt) as a, fm.Problem(R, t, ci, cj, pid, x1, x2, options=opt) as b, \
            fm.Problem(R, t, ci, cj, pid, x1, x2, options=opt) as f:
        for p in (a, b, f):
            p.set_scores(score)
        for r in range(2):       # without a history, then with one
            feats = torch.empty(n, 8, dtype=torch.bfloat16, device="cuda")
            f.collect_features(tau, r, feats)
            p_ref = torch.empty(n, dtype=torch.float32, device="cuda")
            net.forward(feats, p_ref)
            torch.cuda.synchronize()
            e = np.abs(f.residuals().astype(np.float64))
            kept = a.learned_weights(net, tau, cap, r)
            assert kept == int((e <= cap).sum())
            ref = np.where(e <= cap, p_ref.cpu().numpy() / np.maximum(e, 1e-3), 0.0)
            w = a.get_weights()
            tol = 5e-3 / np.maximum(e, 1e-3) + np.abs(ref) * 2.0 ** -11 + 1e-6
            assert (np.abs(w - ref) <= tol).all()
            assert b.step_learned(net, tau, cap, r, 1, count=True) == kept
            assert np.array_equal(b.get_weights(), w)
            a.step(1)
            for u, v in zip(a.get_params(), b.get_params()):
                assert np.array_equal(u, v)
            f.set_params(*a.get_params())
