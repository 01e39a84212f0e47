"""The persistent rotation kernels at the edges of their work split: two cameras, a full and a
just overfull block, more than one summation tree, more cameras than resident warps (the state
then goes through memory), and cameras of more than 32 pairs, against the FP64 oracle.

Tolerances as at ordinary sizes: the initialisation is solved to a relative residual of 1e-9 on
both well-conditioned graphs, so rotations agree to 1e-6; ten Adam steps agree to 1e-3 of a step."""
import numpy as np
import pytest

import oracle as O
from oracle import rotation as G
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


def _graph(n, extra, hub, seed):
    rng = np.random.default_rng(seed)
    pairs = {(k, k + 1) for k in range(n - 1)}
    if hub:
        pairs |= {(0, k) for k in range(1, min(n, 80))}
    for a, b in rng.integers(0, n, (extra, 2)):
        if a != b:
            pairs.add((min(a, b), max(a, b)))
    ci, cj = (np.array(v, np.int32) for v in zip(*sorted(pairs)))
    R = np.stack([O.expmap(rng.normal(size=3)) for _ in range(n)])
    Rrel = np.stack([O.expmap(0.01 * rng.normal(size=3)) @ R[j] @ R[i].T for i, j in zip(ci, cj)])
    return ci, cj, Rrel


@pytest.mark.parametrize("n,extra,hub", [(2, 0, False), (8, 10, False), (9, 10, False), (257, 2000, True),
                                         (1300, 9000, True), (2500, 20000, False)])
def test_initialisation_and_steps(n, extra, hub):
    build.build()
    ci, cj, Rrel = _graph(n, extra, hub, n)
    lr = 1e-3
    with fm.Rotation(ci, cj, Rrel, n, fm.rotation_options(lr=lr)) as rp:
        rp.initialize()
        R0 = rp.rotations()
        assert np.abs(R0 - G.initial_rotations(n, ci, cj, Rrel)).max() < 1e-6
        rp.set_rotations(R0)
        rp.step(4)
        rp.step(0)
        rp.step(5)
        rp.step(1)
        a = rp.params()
        R = rp.rotations()
        rp.set_rotations(R0)
        rp.step(10)
        assert np.array_equal(rp.params(), a)     # the same steps in one launch
    a_o, _ = G.adam(G.six_d_from_rot(R0), ci, cj, Rrel, 10, lr)
    if len(ci) >= n:     # without a cycle every distance is 0 and the geodesic gradient undefined
        assert np.abs(a - a_o).max() < 1e-3 * lr
    else:
        assert np.abs(a - G.six_d_from_rot(R0)).max() <= 10.01 * lr
    np.testing.assert_allclose(R, G.rot_from_6d(a), atol=1e-13)
