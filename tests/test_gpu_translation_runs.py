"""A run advanced alone and among others, bit for bit: items of one run take a kernel of their own (a run alone,
and several where the resident blocks hold an item each), more runs an item the one that reads four at a time,
with 2, 3, 4 and 8 of them at 1,000 cameras and more blocks' worth of items than are resident. Where many
evaluations would be in series (1,000 cameras with 40 pairs each and 8 runs, with 80 and 3 runs; alone: 2 and 3) the
pairs have a phase of their own, in batches of 4 and 2 runs.

Cameras of many pairs (one in all pairs, all in all) take that phase in batches of one run as well: a step of those
against NumPy from the gradient of the evaluation kernels, within 1e-5 of a step (FP32 moments and their quotient:
a few 2^-24; a gradient component that cancels to below 1e-3 of the largest is left out)."""
import numpy as np
import pytest

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


def _directions(rng, n, ci, cj):
    R = np.linalg.qr(rng.normal(size=(n, 3, 3)))[0]
    R *= np.sign(np.linalg.det(R))[:, None, None]
    o = rng.normal(size=(n, 3))
    d = np.einsum("nab,nb->na", R[cj], o[ci] - o[cj])
    return R, d / np.linalg.norm(d, axis=1, keepdims=True)


@pytest.mark.parametrize("n, near, runs", [(5, 2, 3), (90, 40, 4), (1000, 3, 3), (1000, 20, 8), (1000, 40, 3), (1000, 3, 13), (2600, 2, 2)])
def test_runs_do_not_depend_on_each_other(n, near, runs):
    build.build()
    rng = np.random.default_rng(n + runs)
    key = sorted({(min(a, (a + d) % n), max(a, (a + d) % n)) for a in range(n) for d in range(1, near + 1)})
    ci, cj = (np.array(v, np.int32) for v in zip(*key))
    R, d = _directions(rng, n, ci, cj)
    start = rng.normal(size=(runs, n, 3))
    with fm.Translation(R, ci, cj, d, start) as together:
        together.step(7)
        got = together.centres()
    for r in {0, runs // 2, runs - 1}:
        with fm.Translation(R, ci, cj, d, start[r:r + 1]) as alone:
            alone.step(7)
            np.testing.assert_array_equal(alone.centres()[0], got[r])


@pytest.mark.parametrize("runs", [1, 5])
@pytest.mark.parametrize("graph", ["hub", "all"])
def test_cameras_of_many_pairs(graph, runs):
    build.build()
    rng = np.random.default_rng(runs)
    n = 400 if graph == "hub" else 180
    if graph == "hub":
        ci, cj = np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32)
    else:
        ci, cj = (v.astype(np.int32) for v in np.triu_indices(n, 1))
    R, d = _directions(rng, n, ci, cj)
    start = rng.normal(size=(runs, n, 3))
    with fm.Translation(R, ci, cj, d, start) as tr:
        _, grad, _ = tr.loss_grad()
        tr.step(1)
        one = tr.centres()
        tr.step(6)
        got = tr.centres()
        step = (start - one) / 1e-2                      # the first Adam step is the gradient's sign
        sure = np.abs(grad) > 1e-3 * np.abs(grad).max()
        assert np.abs(step[sure] - np.sign(grad[sure])).max() <= 1e-5
        tr.set_centres(start)
        for _ in range(7):
            tr.step(1)
        np.testing.assert_array_equal(tr.centres(), got)
    with fm.Translation(R, ci, cj, d, start[-1:]) as alone:
        alone.step(7)
        np.testing.assert_array_equal(alone.centres()[0], got[-1])
