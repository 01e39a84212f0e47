"""Parameters and poses read back on both sides of the line between one copy and one copy an array (2,048
cameras): what was set, bit for bit, and an error of the device is reported by either."""
import numpy as np
import pytest

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 2047, 2048, 2049, 5000])
def test_parameters_come_back(n):
    build.build()
    rng = np.random.default_rng(n)
    a = rng.uniform(-3, 3, n)
    R = np.stack([np.array([[np.cos(x), 0, np.sin(x)], [0, 1, 0], [-np.sin(x), 0, np.cos(x)]]) for x in a])
    c = rng.normal(size=(n, 3))
    t = -np.einsum("nab,nb->na", R, c)
    ci = np.arange(n - 1, dtype=np.int32)
    x = rng.uniform(-0.5, 0.5, (n - 1, 2)).astype(np.float32)
    with fm.Problem(R, t, ci, ci + 1, ci, x, x) as p:
        p.set_params(R, c)
        for got, want in zip(p.get_params(), (R, c)):
            np.testing.assert_array_equal(got, want)
        got = p.get_poses()
        np.testing.assert_array_equal(got[0], R)
        np.testing.assert_allclose(got[1], t, rtol=0, atol=1e-14)
        c[1] = c[0]                          # a pair without a baseline
        p.set_params(R, c)
        p.step(1)
        with pytest.raises(fm.FastMapError) as e:
            p.get_params()
        assert e.value.status == -4
