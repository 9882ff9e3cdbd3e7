"""The atomic-free spread by block items (widths above 7, and deterministic
plans): every lane split of the widths, samples from far below to above a cell
apart, ragged grids, and column drifts, against the oracle over the full
destination grid; results repeat bit for bit.

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

# n1x, n1y, m2x, m2y, fine cells per sample, heights (um)
GRIDS = {
    "dense": (310, 226, 64, 64, 0.11, 30.0),
    "denser": (700, 90, 64, 64, 0.06, 5.0),
    "half": (150, 146, 64, 128, 0.55, 20.0),
    "one": (94, 130, 128, 128, 1.02, 20.0),
    "sparse": (90, 50, 128, 128, 1.9, 10.0),
    "steep": (100, 100, 128, 128, 1.1, 900.0),
    "sliver": (2, 258, 64, 128, 0.7, 10.0),
}


@functools.lru_cache(maxsize=None)
def case(name):
    n1x, n1y, m2x, m2y, alpha, height = GRIDS[name]
    rng = np.random.default_rng(len(name) + n1x)
    lam, z0, p1 = 633e-9, 0.06, 8e-6
    p2x = alpha * lam * z0 / (p1 * 2 * m2x)
    p2y = alpha * lam * z0 / (p1 * 2 * m2y)
    g = W.geometry(n1x, n1y, p1, p1, m2x, m2y, p2x, p2y, lam, z0)
    d1 = W.surface_smooth_random(g, rng, max(3.0, min(n1x, n1y) / 6), height * 1e-6)
    u1 = W.field_random_amp_phase(g, rng)
    return g, u1, d1, oracle.eq7(g, u1, d1)


@pytest.mark.parametrize("name", list(GRIDS))
@pytest.mark.parametrize("width", [7, 8, 9, 12, 13, 16])
def test_block_spread_matches_oracle(name, width):
    g, u1, d1, ref = case(name)
    with FresnelPlan(g, d1, kernel_width=width, deterministic=width == 7) as plan:
        u = torch.as_tensor(u1, device="cuda")
        a = plan.execute(u)
        b = plan.execute(u)
        torch.cuda.synchronize()
        kind = plan.info()["spread_kind"]
    assert kind in ((2, 4) if width == 7 else (0, 1)), kind
    err = np.linalg.norm(a.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err < max(3.0 * 10.0 ** (-(width - 1)), 5e-6), (name, width, kind, err)
    if kind != 1:
        assert torch.equal(a, b), (name, width, kind)
