"""Direct sums where a term of their phase is no finite number: every sum is a
NaN then, as in FP64 arithmetic, although the phases of Eqs. 5 and 7 are carried
in fixed point, which has no NaN.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import direct_sum  # noqa: E402

pytestmark = pytest.mark.gpu

PTS = (np.arange(10, dtype=np.int32), np.arange(10, dtype=np.int32))


def all_nan(g, u1, d1, form):
    got = direct_sum(g, d1, torch.as_tensor(u1, device="cuda"), form, PTS)
    return bool(torch.isnan(torch.view_as_real(got)).all())


@pytest.mark.parametrize("tilt", [0.0, 0.013])
@pytest.mark.parametrize("height", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("form", [7, 5, 2])
def test_heights(form, height, tilt):
    g, u1, d1 = W.make("sinusoid64")
    d1 = d1.copy()
    d1[5, 63] = height
    assert all_nan(dict(g, sx=tilt, sy=-tilt), u1, d1, form)
    if form == 5:  # destination pitches that differ take a kernel of their own
        assert all_nan(dict(g, sx=tilt, p2y=1.5 * g["p2y"]), u1, d1, form)


@pytest.mark.parametrize("form", [7, 5])
def test_a_sample_in_the_destination_plane(form):
    g, u1, d1 = W.make("sinusoid64")
    d1 = d1.copy()
    d1[63, 0] = g["z0"]
    assert all_nan(g, u1, d1, form)


@pytest.mark.parametrize("form", [7, 5])
def test_an_offset_whose_square_overflows(form):
    g, u1, d1 = W.make("sinusoid64")
    assert all_nan(dict(g, ox=1e200), u1, d1, form)
    assert all_nan(dict(g, oy=1e200), u1, d1, form)
