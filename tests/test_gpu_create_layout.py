"""Problem creation from inputs that are and are not in pair order, at the edges of the layout kernels
(four groups of 32 ahead in the centroid sums, ranges of 2,048, padding), and the refusals that the
focal-length vote finds on the device and its grid's limit. The centroids are fixed-point sums, so the order of the input may
not change a bit: residuals and the initial weights (1) are compared exactly."""
import numpy as np
import pytest

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("sizes", [[2], [31, 1], [127, 1, 1], [1, 128], [2047, 1, 1], [2048, 129], [1] * 300, [700, 5000, 3]])
def test_input_order_changes_no_bit(sizes, storage):
    build.build()
    rng = np.random.default_rng(sum(sizes))
    n_cams = len(sizes) + 1
    a = np.linspace(0.0, 1.0, n_cams)
    R = np.stack([np.array([[np.cos(x), 0, np.sin(x)], [0, 1, 0], [-np.sin(x), 0, np.cos(x)]]) for x in a])
    t = rng.normal(size=(n_cams, 3))
    ci = np.arange(n_cams - 1, dtype=np.int32)
    pid = np.repeat(np.arange(len(sizes), dtype=np.int32), sizes)
    x1, x2 = (rng.uniform(-0.6, 0.6, (len(pid), 2)).astype(np.float32) for _ in range(2))
    perm = rng.permutation(len(pid))
    opt = fm.default_options(storage=storage)
    with fm.Problem(R, t, ci, ci + 1, pid, x1, x2, options=opt) as p:
        e = p.residuals()
        assert p.info()["input_was_sorted"] == 1 and (p.get_weights() == 1).all()
    with fm.Problem(R, t, ci, ci + 1, pid[perm], x1[perm], x2[perm], options=opt) as p:
        assert (p.get_weights() == 1).all()
        np.testing.assert_array_equal(p.residuals(), e[perm])


@pytest.mark.parametrize("n", [1, 63, 64, 65, 700])
def test_focal_vote_names_the_refused_matrix(n):
    build.build()
    F = np.random.default_rng(n).normal(size=(n, 3, 3))
    good = fm.focal_vote(F, [400.0, 500.0], 0.1)
    for value, text in ((0.0, f"F of pair {n - 1} is zero"), (np.nan, "F must be finite"), (np.inf, "F must be finite")):
        B = F.copy()
        B[n - 1] = value
        with pytest.raises(fm.FastMapError, match=text):
            fm.focal_vote(B, [400.0, 500.0], 0.1)
    np.testing.assert_array_equal(fm.focal_vote(F, [400.0, 500.0], 0.1), good)


@pytest.mark.parametrize("n_cand", [65535, 65536, 131071])
def test_focal_vote_with_more_candidates_than_rows_of_blocks(n_cand):
    # every candidate list repeats the same 7 values: equal candidates get equal bits in any block
    build.build()
    F = np.random.default_rng(1).normal(size=(257, 3, 3))
    c = np.resize(np.linspace(300.0, 900.0, 7), n_cand)
    few = fm.focal_vote(F, c[:7], 0.1)
    np.testing.assert_array_equal(fm.focal_vote(F, c, 0.1), np.resize(few, n_cand))
