"""Direct sums at the edges of their fixed-point phases and their split.

Samples are dealt to blocks of 256 threads and points to groups of 8, so the
sizes below leave ragged ends of both; destination indices outside the grid
(also negative) and unequal destination pitches take the phase products
through their whole range.  Tolerance: as in test_gpu_direct, 2e-6 relative
to the FP64 oracle (FP32 products and outputs).
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import direct_sum  # noqa: E402

pytestmark = pytest.mark.gpu

ORACLE = {7: oracle.eq7, 5: oracle.eq5, 2: oracle.eq2}


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("form", [7, 5, 2])
@pytest.mark.parametrize("n1x,n1y,points,p2y", [(2, 2, 1, 9e-6), (34, 22, 9, 9e-6),
                                                (130, 514, 129, 6e-6), (1202, 910, 3, 9e-6)])
def test_direct_sum_ragged(form, n1x, n1y, points, p2y):
    rng = np.random.default_rng(n1x + points + form)
    g = W.geometry(n1x, n1y, 8e-6, 6e-6, 256, 128, 9e-6, p2y, 532e-9, 0.15)
    d1 = rng.uniform(-2e-4, 2e-4, (n1y, n1x))
    u1 = W.field_random_amp_phase(g, rng)
    pts = (rng.integers(-300, 600, points).astype(np.int32),
           rng.integers(-300, 600, points).astype(np.int32))
    got = direct_sum(g, d1, torch.as_tensor(u1, device="cuda"), form, pts).cpu().numpy()
    assert rel_l2(got, ORACLE[form](g, u1, d1, points=pts)) < 2e-6


@pytest.mark.parametrize("form", [7, 5, 2])
def test_direct_sum_keeps_nan_heights(form):
    """Heights are not checked here: a NaN makes every sum a NaN."""
    g, u1, d1 = W.make("sinusoid64")
    d1 = d1.copy()
    d1[63, 63] = np.nan
    pts = (np.arange(10, dtype=np.int32), np.arange(10, dtype=np.int32))
    got = direct_sum(g, d1, torch.as_tensor(u1, device="cuda"), form, pts)
    assert torch.isnan(torch.view_as_real(got)).all()
