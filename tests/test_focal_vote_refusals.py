"""Refused arguments of the focal-length vote, without a usable device: a fundamental matrix that is not finite
or is zero is reported as such, before the arguments behind it and before the missing device."""
import numpy as np
import pytest

import paper_2605_18052_gb300 as fm
from paper_2605_18052_gb300 import build


def _refused(F, cand=(400.0, 500.0), **known):
    build.build()
    with pytest.raises(fm.FastMapError) as e:
        fm.focal_vote(F, list(cand), 0.1, **known)
    return e.value.status, str(e.value)


def test_refused_matrix_comes_first():
    F = np.random.default_rng(0).normal(size=(70, 3, 3))
    for value, at, text in ((np.nan, 69, "F must be finite"), (np.inf, 0, "F must be finite"), (0.0, 64, "F of pair 64 is zero")):
        B = F.copy()
        B[at] = value
        for kw in (dict(), dict(cand=(0.0, 500.0)), dict(f1_known=np.full(70, -1.0)), dict(f2_known=np.full(70, np.nan))):
            status, msg = _refused(B, **kw)
            assert status == -1 and text in msg
    B = F.copy()
    B[3], B[60] = 0.0, np.nan       # the first refused matrix decides
    assert "F of pair 3 is zero" in _refused(B)[1]


def test_other_arguments_are_refused_with_good_matrices():
    F = np.random.default_rng(1).normal(size=(3, 3, 3))
    assert "candidates" in _refused(F, cand=(np.nan,))[1]
    assert "known focal lengths" in _refused(F, f1_known=np.array([0.0, -1.0, 2.0]))[1]
