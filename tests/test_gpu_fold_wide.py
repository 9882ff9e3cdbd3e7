"""Widths above 7 on folding and wrapping maps (2 or 4 lanes share a source
column; at odd widths the last lane has taps to leave out), at ragged grids,
against the oracle over the full destination grid.

Tolerance as in test_kernel_width_accuracy: the kernel width's truncation, or
5e-6 for FP32 rounding.
"""
from __future__ import annotations

import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402

pytestmark = pytest.mark.gpu

# n1x, n1y, m2x, m2y, fine cells per sample, heights (um), random heights
GRIDS = {
    "wrapping": (150, 94, 64, 64, 1.3, 30.0, False),
    "wrapping_y": (50, 290, 128, 64, 0.9, 20.0, False),
    "folding": (94, 130, 64, 128, 0.6, 3000.0, True),
    "sliver": (2, 258, 64, 64, 0.9, 10.0, False),
}


@functools.lru_cache(maxsize=None)
def case(name):
    n1x, n1y, m2x, m2y, alpha, height, rough = GRIDS[name]
    rng = np.random.default_rng(n1x + n1y)
    lam, z0, p1 = 633e-9, 0.06, 8e-6
    p2x = alpha * lam * z0 / (p1 * 2 * m2x)
    p2y = alpha * lam * z0 / (p1 * 2 * m2y)
    g = W.geometry(n1x, n1y, p1, p1, m2x, m2y, p2x, p2y, lam, z0)
    d1 = (rng.uniform(-0.5, 0.5, (n1y, n1x)) if rough
          else W.surface_smooth_random(g, rng, max(3.0, min(n1x, n1y) / 6), 1.0)) * height * 1e-6
    u1 = W.field_random_amp_phase(g, rng)
    return g, u1, d1, oracle.eq7(g, u1, d1)


@pytest.mark.parametrize("name", list(GRIDS))
@pytest.mark.parametrize("width", [8, 9, 12, 13, 16])
def test_fold_spread_matches_oracle(name, width):
    g, u1, d1, ref = case(name)
    with FresnelPlan(g, d1, kernel_width=width) as plan:
        out = plan.execute(torch.as_tensor(u1, device="cuda")).cpu().numpy()
        assert plan.info()["spread_kind"] == 1
    err = np.linalg.norm(out - ref) / np.linalg.norm(ref)
    assert err < max(3.0 * 10.0 ** (-(width - 1)), 5e-6), (name, width, err)
