"""asfd_plan_update_d1 has finished when it returns: the new height map may be
used on any stream at once, and the heights' buffer reused."""
from __future__ import annotations

import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(), dict(deterministic=True), dict(kind="learned")],
                         ids=["default", "repeatable", "learned"])
def test_nothing_is_left_on_the_stream(kw):
    m = 512
    lam, z0, p1 = 633e-9, 0.06, 1e-6
    p2 = 0.05 * lam * z0 / (p1 * 2 * m)
    g = W.geometry(16384, 4096, p1, p1, m, m, p2, p2, lam, z0)
    d1 = torch.zeros((4096, 16384), dtype=torch.float64, device="cuda")
    other = torch.full_like(d1, 1e-5)
    s = torch.cuda.Stream()
    with FresnelPlan(g, d1, **kw) as plan:
        torch.cuda.synchronize()
        for heights in (other, d1, other, d1):
            plan.update_d1(heights, stream=s)
            assert s.query()
