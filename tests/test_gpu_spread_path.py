"""Which spread a plan takes (asfd_debug_spread_path): the rules of the dispatch at
sizes where a change of one of them would go unseen in the results."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import capi, workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402

pytestmark = pytest.mark.gpu

WRAPPED, ITEM_TILES, BLOCK_ITEMS = 1, 4, 5


def spread_path(plan):
    """(path, warps, chunks, rows, dup)"""
    out = (ctypes.c_int * 5)()
    capi._check(capi.load().asfd_debug_spread_path(plan.handle, out))
    return tuple(out)


@pytest.mark.parametrize("n", [32, 64, 96])
@pytest.mark.parametrize("alpha", [1.03, 1.5])
def test_small_repeatable_plans_take_item_tiles(n, alpha):
    """Tiny grids have shorter runs in the default spread, not in the item tiles."""
    lam, z0, p1, m = 633e-9, 0.06, 8e-6, 128
    p2 = alpha * lam * z0 / (p1 * 2 * m)
    g = W.geometry(n, n, p1, p1, m, m, p2, p2, lam, z0)
    with FresnelPlan(g, np.zeros((n, n)), deterministic=True) as plan:
        assert spread_path(plan)[0] == ITEM_TILES
