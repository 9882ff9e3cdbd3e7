"""What a plan holds per source sample: its q (4 bytes).  The q of a height map being
checked waits in a work buffer where there is one, and a rejected map changes nothing
wherever it waited.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import capi, workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402

pytestmark = pytest.mark.gpu


def test_bytes_per_sample():
    n, m = 1024, 512
    g = W.geometry(n, n, 8e-6, 8e-6, m, m, 1e-6, 1e-6, 633e-9, 0.06)
    u = torch.ones((n, n), dtype=torch.complex64, device="cuda")
    with FresnelPlan(g, np.zeros((n, n))) as plan:
        # q and 1/256 of a source tile's tables; the axis tables are O(n)
        created = plan.info()["device_bytes"]
        assert created < 4.5 * n * n + 400 * n
        plan.execute(u)
        work = plan.info()["device_bytes"]
        plan.update_d1(np.full((n, n), 1e-5))
        assert plan.info()["device_bytes"] == work
    with FresnelPlan(g, np.zeros((n, n)), workspace=True) as plan:
        plan.update_d1(np.full((n, n), 1e-5))
        assert plan.info()["device_bytes"] == created


@pytest.mark.parametrize("m", [64, 512])
@pytest.mark.parametrize("before", ["nothing", "execute", "workspace"])
def test_a_rejected_map_leaves_the_plan_as_it_was(before, m):
    """m = 64: the row buffer is too small for q (512 x 512 samples)."""
    rng = np.random.default_rng(m)
    n = 512
    p2 = 0.2 * 633e-9 * 0.06 / (8e-6 * 2 * m)
    g = W.geometry(n, n, 8e-6, 8e-6, m, m, p2, p2, 633e-9, 0.06)
    d1 = W.surface_smooth_random(g, rng, 20.0, 10e-6)
    u = torch.as_tensor(W.field_random_amp_phase(g, rng), device="cuda")
    with FresnelPlan(g, d1, deterministic=True) as plan:
        want = plan.execute(u)
    with FresnelPlan(g, d1 + 1e-5, deterministic=True, workspace=before == "workspace") as plan:
        if before == "execute":
            plan.execute(u)
        plan.update_d1(d1)
        assert torch.equal(plan.execute(u), want)
        for bad in (np.nan, np.inf, g["z0"], 0.2 * g["z0"]):
            worse = d1 + 1e-5
            worse[7, 9] = bad
            with pytest.raises(capi.AsfdError):
                plan.update_d1(worse)
            assert torch.equal(plan.execute(u), want)
