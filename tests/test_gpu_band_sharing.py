"""Spreads that add into a zero band (widths above 7, folding and wrapping maps,
block items of deterministic plans) where something other than the plan's own
calls has written the fine grid since: another plan of the same workspace, and
replays of a captured call.

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

# width, deterministic, fine cells per sample, height (um); 256 samples on 128
# points wrap from one cell per sample on
CASES = {
    "wide": (12, False, 0.7, 10.0),
    "wide_wrapping": (12, False, 1.3, 10.0),
    "window_wrapping": (7, False, 1.3, 10.0),
    "repeatable": (7, True, 0.7, 10.0),
}


def make(name, n=256, m=128, seed=5):
    width, det, alpha, height = CASES[name]
    lam, z0, p1 = 633e-9, 0.06, 8e-6
    p2 = alpha * lam * z0 / (p1 * 2 * m)
    g = W.geometry(n, n, p1, p1, m, m, p2, p2, lam, z0)
    rng = np.random.default_rng(seed)
    d1 = W.surface_smooth_random(g, rng, 20.0, height * 1e-6)
    u1 = torch.as_tensor(W.field_random_amp_phase(g, rng), device="cuda")
    return FresnelPlan(g, d1, kernel_width=width, deterministic=det), u1


def close(a, b):
    return float((a - b).norm() / b.norm()) < 1e-6


@pytest.mark.parametrize("name", list(CASES))
def test_plans_that_share_a_workspace(name):
    a, ua = make(name)
    b, ub = make(name, n=200, m=128, seed=6)
    with a, b:
        want_a, want_b = a.execute(ua), b.execute(ub)
        ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
        a.set_workspace(ws)
        b.set_workspace(ws)
        for _ in range(2):
            assert close(a.execute(ua), want_a)
            ws.fill_(64)  # the owner uses it between calls (3.0 as floats)
            assert close(b.execute(ub), want_b)
            ws.fill_(64)
        a.set_workspace(None)
        b.set_workspace(None)


@pytest.mark.parametrize("name", list(CASES))
def test_calls_between_replays(name):
    plan, u = make(name)
    with plan:
        want = plan.execute(u)
        gu = torch.randn_like(want)
        g1 = torch.empty_like(u)
        out = torch.empty_like(want)
        plan.adjoint(None, gu, g1, None)
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        fwd, adj = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(fwd, stream=s):
            plan.execute(u, out)
        with torch.cuda.graph(adj, stream=s):
            plan.adjoint(None, gu, g1, None)
        torch.cuda.current_stream().wait_stream(s)
        for _ in range(2):
            adj.replay()
            assert close(plan.execute(u), want)
            adj.replay()
            fwd.replay()
            assert close(out, want)
            plan.adjoint(None, gu, g1, None)
            fwd.replay()
            assert close(out, want)
