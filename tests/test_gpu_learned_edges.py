"""Gradients of the learned kernel where its kernels have ragged ends: source
tiles cut by the grid's edge, tile counts that are no multiple of a group,
destinations wider than one block's columns, footprints that wrap around the
fine grid; and fields so faint that squares leave FP32's range.

Directional derivatives against central differences of the CPU model (tests'
tolerance for the gradient, 3e-3: FP32 gradients, differences of step 1e-4).
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import learned_ref as R  # noqa: E402
from paper_1203_3583_gb300 import capi, workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402
from tests.test_gpu_learned import _perturbed_params  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    "ragged": W.geometry(50, 38, 10e-6, 7e-6, 64, 32, 12e-6, 9e-6, 532e-9, 0.04),
    "wide": W.geometry(150, 70, 6e-6, 9e-6, 256, 64, 5e-6, 9e-6, 633e-9, 0.05),
    "wrapping": W.geometry(64, 34, 20e-6, 20e-6, 64, 64, 20e-6, 20e-6, 633e-9, 0.02),
}


def _gradient(name, scale=1.0):
    rng = np.random.default_rng(71)
    g = CASES[name]
    d1 = W.surface_smooth_random(g, rng, 5.0, 40e-6)
    u1 = (rng.standard_normal(d1.shape) + 1j * rng.standard_normal(d1.shape)).astype(np.complex64)
    # a target well away from the model's output, so that the residual is no rounding
    target = (oracle.eq7(g, u1, d1) * (1 + 0.3 * rng.standard_normal((g["m2y"], g["m2x"])))).astype(np.complex64)
    with FresnelPlan(g, d1, kind="learned") as plan:
        params = _perturbed_params(plan, 72)
        grad, loss = capi.asfd_learned_gradient(
            plan.handle, torch.as_tensor(u1 * np.float32(scale), device="cuda"),
            torch.as_tensor(target * np.float32(scale), device="cuda"), plan.shape1, plan.shape2)
    return g, u1, d1, target, params, grad.astype(np.float64), loss


@pytest.mark.parametrize("name", list(CASES))
def test_directional_derivatives(name):
    g, u1, d1, target, params, grad, loss = _gradient(name)
    assert abs(loss - R.loss(R.forward(g, u1, d1, params), target)) < 1e-4 * loss
    rng = np.random.default_rng(73)
    for sl in (R.SL_BASE, R.SL_W1, R.SL_B1, R.SL_W2, R.SL_B2, R.SL_DX, R.SL_DY):
        v = np.zeros_like(params)
        v[sl] = grad[sl] / np.linalg.norm(grad[sl]) + 0.1 * rng.standard_normal(sl.stop - sl.start) / np.sqrt(sl.stop - sl.start)
        h = 1e-4 * max(1.0, float(np.abs(params[sl]).max()))
        fd = (R.loss(R.forward(g, u1, d1, params + h * v), target) -
              R.loss(R.forward(g, u1, d1, params - h * v), target)) / (2 * h)
        assert abs(fd - grad @ v) < 3e-3 * np.linalg.norm(grad[sl]), (name, sl)


def test_faint_fields():
    """The relative loss does not depend on the fields' scale; 2^-50 is exact."""
    a = _gradient("ragged")
    b = _gradient("ragged", 2.0 ** -50)
    assert abs(a[6] - b[6]) < 1e-6 * a[6]
    assert np.linalg.norm(a[5] - b[5]) < 1e-5 * np.linalg.norm(a[5])
