"""A run advanced alone and among others, bit for bit: items of one run take a kernel of their own (a run alone,
and several where the resident blocks hold an item each), more runs an item the one that reads four at a time,
with 2, 3, 4 and 8 of them at 1,000 cameras and more blocks' worth of items than are resident."""
import numpy as np
import pytest

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, near, runs", [(5, 2, 3), (90, 40, 4), (1000, 3, 3), (1000, 20, 8), (1000, 3, 13), (2600, 2, 2)])
def test_runs_do_not_depend_on_each_other(n, near, runs):
    build.build()
    rng = np.random.default_rng(n + runs)
    key = sorted({(min(a, (a + d) % n), max(a, (a + d) % n)) for a in range(n) for d in range(1, near + 1)})
    ci, cj = (np.array(v, np.int32) for v in zip(*key))
    R = np.linalg.qr(rng.normal(size=(n, 3, 3)))[0]
    R *= np.sign(np.linalg.det(R))[:, None, None]
    o = rng.normal(size=(n, 3))
    d = np.einsum("nab,nb->na", R[cj], o[ci] - o[cj])
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    start = rng.normal(size=(runs, n, 3))
    with fm.Translation(R, ci, cj, d, start) as together:
        together.step(7)
        got = together.centres()
    for r in {0, runs // 2, runs - 1}:
        with fm.Translation(R, ci, cj, d, start[r:r + 1]) as alone:
            alone.step(7)
            np.testing.assert_array_equal(alone.centres()[0], got[r])
