"""Which spread a plan takes (asfd_debug_spread_path): the rules of the dispatch at
sizes where a change of one of them would go unseen in the results."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1203_3583_gb300 import capi, workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402
from tests.test_gpu_spread_block import GRIDS, case  # noqa: E402

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


# (grid of test_gpu_spread_block, width): the block's shape is checked where it is the point
BLOCK = [(name, w) for name in GRIDS for w in (8, 9, 12, 13, 16)] + \
        [(name, 7) for name in ("dense", "denser", "half", "sliver")]


@pytest.mark.parametrize("name,width", BLOCK)
def test_block_items(name, width):
    """Monotone maps at widths above 7, and repeatable plans whose samples are less
    than a cell apart: block items, the oracle's field and equal bits in two runs."""
    g, u1, d1, ref = case(name)
    with FresnelPlan(g, d1, kernel_width=width, deterministic=width == 7) as plan:
        path, warps, chunks, rows, dup = spread_path(plan)
        u = torch.as_tensor(u1, device="cuda")
        a = plan.execute(u)
        b = plan.execute(u)
        torch.cuda.synchronize()
    assert path == BLOCK_ITEMS
    assert dup == (1 if GRIDS[name][4] < 1.0 else 0)
    if name == "denser" and width > 7:  # blocks two apart meet unless warps take chunks in turn
        assert warps == 8 and chunks > 1
    assert torch.equal(a, b)
    err = np.linalg.norm(a.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err < max(3.0 * 10.0 ** (-(width - 1)), 5e-6), (name, width, err)


@pytest.mark.parametrize("width", [7, 8, 16])
@pytest.mark.parametrize("deterministic", [False, True])
def test_wrapping_maps_take_wrapped_windows(width, deterministic):
    lam, z0, p1, m, n = 633e-9, 0.06, 8e-6, 64, 150
    p2 = 1.3 * lam * z0 / (p1 * 2 * m)
    g = W.geometry(n, n, p1, p1, m, m, p2, p2, lam, z0)
    with FresnelPlan(g, np.zeros((n, n)), kernel_width=width, deterministic=deterministic) as plan:
        assert spread_path(plan)[0] == WRAPPED


CONFLICT_FREE, SLIDING = 0, 2


@pytest.mark.parametrize("width,deterministic,sparse", [(4, True, 2.5), (7, True, 2.5), (8, False, 4.0),
                                                        (12, False, 6.0), (14, False, 7.0)])
@pytest.mark.parametrize("ratio", [1.0, 2.0])
def test_sparse_maps_take_conflict_free_tiles(width, deterministic, sparse, ratio):
    """Fine cells per sample on both sides of the line (their product counts), and the
    oracle's field there."""
    lam, z0, p1, n = 633e-9, 0.06, 8e-6, 44
    rng = np.random.default_rng(width)
    for cells, paths in ((0.93 * sparse, (ITEM_TILES, BLOCK_ITEMS)),
                         (1.07 * sparse, (ITEM_TILES, SLIDING if width <= 7 else CONFLICT_FREE))):
        ax, ay = np.sqrt(cells * ratio), np.sqrt(cells / ratio)
        m = 128
        g = W.geometry(n, n, p1, p1, m, m, ax * lam * z0 / (p1 * 2 * m), ay * lam * z0 / (p1 * 2 * m),
                       lam, z0)
        d1 = W.surface_smooth_random(g, rng, 8.0, 10e-6)
        u1 = W.field_random_amp_phase(g, rng)
        with FresnelPlan(g, d1, kernel_width=width, deterministic=deterministic) as plan:
            path = spread_path(plan)[0]
            out = plan.execute(torch.as_tensor(u1, device="cuda")).cpu().numpy()
        assert path in (paths if width <= 7 else paths[1:]), (cells, path)
        ref = oracle.eq7(g, u1, d1)
        err = np.linalg.norm(out - ref) / np.linalg.norm(ref)
        assert err < max(3.0 * 10.0 ** (-(width - 1)), 5e-6), (cells, path, err)
