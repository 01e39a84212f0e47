"""The initialisation of graphs with cameras of many pairs, against the FP64 oracle: 256 and 257 pairs (the line
from which the next pairs are read ahead), all pairs, one camera in all pairs.

Tolerance as at ordinary sizes: solved to a relative residual of 1e-9 on well-conditioned graphs, so rotations
agree to 1e-6."""
import numpy as np
import pytest

import oracle as O
from oracle import rotation as G
import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, hub, extra", [(257, 0, 0), (258, 0, 0), (300, 256, 900), (300, 257, 900), (400, 399, 0)])
def test_initialisation(n, hub, extra):
    build.build()
    rng = np.random.default_rng(n + hub)
    if hub == 0:
        pairs = {(a, b) for a in range(n) for b in range(a + 1, n)}
    else:
        pairs = {(k, k + 1) for k in range(n - 1)} | {(min(3, k), max(3, k)) for k in range(hub + 1) if k != 3}
        pairs |= {(min(a, b), max(a, b)) for a, b in rng.integers(4, n, (extra, 2)) if a != b}
    ci, cj = (np.array(v, np.int32) for v in zip(*sorted(pairs)))
    R = np.stack([O.expmap(rng.normal(size=3)) for _ in range(n)])
    noise = np.stack([O.expmap(0.01 * v) for v in rng.normal(size=(len(ci), 3))])
    Rrel = noise @ R[cj] @ R[ci].transpose(0, 2, 1)
    with fm.Rotation(ci, cj, Rrel, n) as rp:
        rp.initialize()
        got = rp.rotations()
        rp.initialize()
        np.testing.assert_array_equal(rp.rotations(), got)
    assert np.abs(got - G.initial_rotations(n, ci, cj, Rrel)).max() < 1e-6
