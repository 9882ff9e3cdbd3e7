"""Captured calls replayed after the plan's height map has changed: with the shape
that they were captured with they transform a map that differs a little, and stay
inside their own buffers whatever the map is.

Tolerance: two evaluations differ by the order of float additions only (1e-6
relative L2, as in test_run_twice).
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402

pytestmark = pytest.mark.gpu

# width, deterministic, fine cells per sample, samples, destination points
CASES = {
    "default": (7, False, 0.7, 256, 128),
    "wide": (12, False, 1.04, 256, 256),
    "widest": (16, False, 0.7, 200, 128),
    "repeatable_close": (7, True, 0.7, 256, 128),
    "repeatable": (7, True, 1.04, 256, 256),
    "wrapping": (12, False, 1.3, 256, 128),
}


def geometry(name):
    width, det, alpha, n, m = CASES[name]
    lam, z0, p1 = 633e-9, 0.06, 8e-6
    p2 = alpha * lam * z0 / (p1 * 2 * m)
    return W.geometry(n, n, p1, p1, m, m, p2, p2, lam, z0), dict(kernel_width=width, deterministic=det)


def fresh(g, d1, u, kw):
    with FresnelPlan(g, d1, **kw) as plan:
        return plan.execute(u)


def close(a, b):
    return float((a - b).norm() / b.norm()) < 1e-6


def captured(plan, u, out):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        plan.execute(u, out)
    torch.cuda.current_stream().wait_stream(s)
    return graph


# (item tiles take the boxes of the map as they are, without room for others)
@pytest.mark.parametrize("name", [n for n in CASES if n != "repeatable"])
def test_small_changes(name):
    g, kw = geometry(name)
    rng = np.random.default_rng(8)
    base = W.surface_smooth_random(g, rng, 20.0, 10e-6)
    u = torch.as_tensor(W.field_random_amp_phase(g, rng), device="cuda")
    with FresnelPlan(g, base, **kw) as plan:
        out = torch.empty_like(plan.execute(u))
        graph = captured(plan, u, out)
        band = [plan.info()[k] for k in ("band_x0", "band_x1", "band_y0", "band_y1")]
        for _ in range(6):
            d1 = base + W.surface_smooth_random(g, rng, 20.0, 10e-6)
            plan.update_d1(d1)
            assert [plan.info()[k] for k in ("band_x0", "band_x1", "band_y0", "band_y1")] == band
            graph.replay()
            want = fresh(g, d1, u, kw)
            assert close(out, want)
            assert close(plan.execute(u), want)


@pytest.mark.parametrize("name", list(CASES))
def test_large_changes(name):
    """Replays on a map that the launch was not made for give no promise about their
    output; the plan's own calls are right before and after, and a new capture is."""
    g, kw = geometry(name)
    rng = np.random.default_rng(9)
    u = torch.as_tensor(W.field_random_amp_phase(g, rng), device="cuda")
    maps = [W.surface_smooth_random(g, rng, 20.0, 10e-6), W.surface_smooth_random(g, rng, 60.0, 5e-3),
            np.full((g["n1y"], g["n1x"]), -5e-3), np.full((g["n1y"], g["n1x"]), 5e-3),
            W.surface_smooth_random(g, rng, 3.0, 100e-6)]
    with FresnelPlan(g, maps[0], **kw) as plan:
        out = torch.empty_like(plan.execute(u))
        graphs = [captured(plan, u, out)]
        for d1 in maps[1:] + maps[:1]:
            plan.update_d1(d1)
            want = fresh(g, d1, u, kw)
            assert close(plan.execute(u), want)
            for graph in graphs:
                graph.replay()
            assert close(plan.execute(u), want)
            graphs.append(captured(plan, u, out))
            graphs[-1].replay()
            assert close(out, want)
