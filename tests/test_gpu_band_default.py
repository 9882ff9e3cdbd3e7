"""The default spread adds into a zero band that the row pass before has left:
also where something other than the plan's own calls has written the fine grid
since (another plan of the same workspace, replays of captured calls, a sum over
surfaces, a batch).

Tolerance as in test_gpu_band_sharing: two evaluations differ by the order of
float additions only (1e-6 relative L2).
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan, multi_execute  # noqa: E402

pytestmark = pytest.mark.gpu

KINDS = ["es", "learned"]


def case(n=256, m=128, alpha=0.7, seed=5):
    lam, z0, p1 = 633e-9, 0.06, 8e-6
    p2 = alpha * lam * z0 / (p1 * 2 * m)
    g = W.geometry(n, n, p1, p1, m, m, p2, p2, lam, z0)
    rng = np.random.default_rng(seed)
    d1 = W.surface_smooth_random(g, rng, 20.0, 10e-6)
    return g, d1, torch.as_tensor(W.field_random_amp_phase(g, rng), device="cuda")


def make(kind, **k):
    g, d1, u1 = case(**k)
    return FresnelPlan(g, d1, kind=kind), u1


def close(a, b):
    return float((a - b).norm() / b.norm()) < 1e-6


def adjoint(plan, grad):
    plan.adjoint(None, grad, torch.empty(plan.shape1, dtype=torch.complex64, device="cuda"), None)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("m", [128, 64])
def test_plans_that_share_a_workspace(kind, m):
    """A plan's grid holds the other's adjoint grid, or its row buffer."""
    a, ua = make(kind)
    b, ub = make(kind, n=160, m=m, seed=6)
    with a, b:
        want_a, want_b = a.execute(ua), b.execute(ub)
        ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
        a.set_workspace(ws)
        b.set_workspace(ws)
        for _ in range(2):
            assert close(a.execute(ua), want_a)
            adjoint(b, want_b)
            assert close(a.execute(ua), want_a)
            assert close(b.execute(ub), want_b)
        a.set_workspace(None)
        b.set_workspace(None)


def captured(call):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call()
    torch.cuda.current_stream().wait_stream(s)
    return g


@pytest.mark.parametrize("kind", KINDS)
def test_calls_between_replays(kind):
    plan, u = make(kind)
    with plan:
        want = plan.execute(u)
        out, g1 = torch.empty_like(want), torch.empty_like(u)
        plan.adjoint(None, want, g1, None)
        want_g1 = g1.clone()
        plan.execute(u)
        adj = captured(lambda: plan.adjoint(None, want, g1, None))
        both = captured(lambda: (plan.execute(u, out), plan.adjoint(None, want, g1, None)))
        for _ in range(2):
            adj.replay()
            assert close(plan.execute(u), want)
            both.replay()
            assert close(out, want) and close(g1, want_g1)
            both.replay()
            assert close(out, want)
            assert close(plan.execute(u), want)


def test_a_first_call_that_is_captured():
    """Capturing runs nothing: the band is as dirty after it as before."""
    plan, u = make("es")
    with plan:
        want = plan.execute(u)
        out = torch.empty_like(want)
        adjoint(plan, want)
        fwd = captured(lambda: plan.execute(u, out))
        assert close(plan.execute(u), want)
        fwd.replay()
        assert close(out, want)


def test_a_captured_sum_over_surfaces():
    a, ua = make("es")
    b, ub = make("es", seed=6)
    with a, b:
        want = a.execute(ua)
        total = multi_execute([a, b], [ua, ub])
        out = torch.empty_like(total)
        adjoint(a, want)
        g = captured(lambda: multi_execute([a, b], [ua, ub], out))
        assert close(a.execute(ua), want)
        g.replay()
        assert close(out, total)
        assert close(a.execute(ua), want)
