"""The persistent translation kernel at the edges of its work split: two cameras, a full and a
just overfull block, run counts around the batch and item sizes, more items than resident blocks
(the state then goes through memory) and cameras of more than 32 pairs. A launch of ten iterations
must equal launches of one, three and six bit for bit. Each of three single iterations is compared
with an Adam step in NumPy from the gradient that the evaluation kernels give at the same centres
(the oracle's test covers those): the FP32 moments are a few roundings, so the step agrees to 1e-5 of the
step size."""
import numpy as np
import pytest

import oracle as O
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,runs,extra,hub", [(2, 1, 0, False), (8, 4, 12, False), (9, 5, 12, True), (50, 9, 200, True),
                                              (700, 8, 3000, True), (2600, 3, 9000, False)])
def test_steps_at_the_edges(n, runs, extra, hub):
    build.build()
    rng = np.random.default_rng(n)
    pairs = {(k, k + 1) for k in range(n - 1)}
    if hub:
        pairs |= {(0, k) for k in range(1, min(n, 80))}
    pairs |= {(min(a, b), max(a, b)) for a, b in rng.integers(0, n, (extra, 2)) if a != b}
    ci, cj = (np.array(v, np.int32) for v in zip(*sorted(pairs)))
    R = np.stack([O.expmap(rng.normal(size=3)) for _ in range(n)])
    t = rng.normal(size=(len(ci), 3))
    t /= np.linalg.norm(t, axis=1, keepdims=True)
    o0 = rng.normal(size=(runs, n, 3))
    lr = 1e-2
    with fm.Translation(R, ci, cj, t, o0, fm.translation_options(lr=lr)) as tr:
        for k in (1, 0, 3, 6):
            tr.step(k)
        a = tr.centres()
        tr.set_centres(o0)
        tr.step(10)
        assert np.array_equal(tr.centres(), a)
        tr.set_centres(o0)
        m, v = np.zeros_like(o0), np.zeros_like(o0)
        for k in range(1, 4):
            before, g = tr.centres(), tr.loss_grad()[1].astype(np.float32).astype(np.float64)
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            step = lr * (m / (1 - 0.9 ** k)) / (np.sqrt(v / (1 - 0.999 ** k)) + 1e-12)
            tr.step(1)
            assert np.abs(before - step - tr.centres()).max() <= 1e-5 * lr + 1e-15
