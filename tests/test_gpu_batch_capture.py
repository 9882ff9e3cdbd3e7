"""A batch whose first call is captured into a graph of the caller's: capturing
runs nothing, so the bands that its spreads add into are not clean after it.
Tolerance as in test_gpu_band_sharing (the order of float additions)."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelBatch, FresnelPlan  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,alpha", [(7, 0.7), (8, 0.7), (8, 1.3)])
def test_first_call_captured(width, alpha):
    items, u1s, want = [], [], []
    for seed in (5, 6, 7):
        m = 64 * 2 ** (seed - 5)
        p2 = alpha * 633e-9 * 0.06 / (8e-6 * 2 * m)
        g = W.geometry(2 * m, 2 * m, 8e-6, 8e-6, m, m, p2, p2, 633e-9, 0.06)
        rng = np.random.default_rng(seed)
        d1 = W.surface_smooth_random(g, rng, 20.0, 10e-6)
        u = torch.as_tensor(W.field_random_amp_phase(g, rng), device="cuda")
        with FresnelPlan(g, d1, kernel_width=width) as p:
            want.append(p.execute(u))
        items.append((g, d1))
        u1s.append(u)
    outs = [torch.empty_like(w) for w in want]
    with FresnelBatch(items, kernel_width=width) as batch:
        # (the persistent kernel leaves the bands as its rows were read; the stream
        # schedule starts over after it)
        batch.set_schedule("persistent")
        batch.execute(u1s)
        batch.set_schedule("streams")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            batch.execute(u1s, outs)
        torch.cuda.current_stream().wait_stream(s)
        for _ in range(3):
            got = batch.execute(u1s)
            graph.replay()
            for a, b, w in zip(got, outs, want):
                assert float((a - w).norm() / w.norm()) < 1e-6
                assert float((b - w).norm() / w.norm()) < 1e-6
