"""The adjoint's interpolation at even and odd widths (their cells are read in
pairs from an even column, with masks that differ), with and without wrapped
footprints, at ragged sizes.

Gradients against the oracle's, with the width's truncation (test_kernel_width_accuracy)
or the bounds of test_gradients_match_oracle (1e-5 and 1e-4); the height gradient takes
the kernel's derivative, tenfold the truncation.  At widths 2 and 4, whose truncation
says little, the dot-product identity with the forward transform (FP32 rounding) shows
that every tap is the forward's.
"""
from __future__ import annotations

import functools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402
from tests.test_gpu_adjoint import crandn, gpu_adjoint, rel_l2  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    "ragged": W.geometry(50, 38, 10e-6, 7e-6, 64, 32, 12e-6, 9e-6, 532e-9, 0.04),
    "wrapping": W.geometry(66, 34, 20e-6, 20e-6, 64, 64, 20e-6, 20e-6, 633e-9, 0.02),
}


@functools.lru_cache(maxsize=None)
def case(name):
    rng = np.random.default_rng(41)
    g = CASES[name]
    u1 = crandn(rng, (g["n1y"], g["n1x"]))
    d1 = W.surface_smooth_random(g, rng, 4.0, 60e-6) - 30e-6
    gu2 = crandn(rng, (g["m2y"], g["m2x"]))
    return g, u1, d1, gu2, oracle.eq7_grad(g, u1, d1, gu2)


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("width", [2, 3, 4, 6, 7, 8, 13, 15])
def test_gradients(name, width):
    g, u1, d1, gu2, (ref_u1, ref_d1) = case(name)
    with FresnelPlan(g, d1, kernel_width=width) as plan:
        fwd = plan.execute(torch.as_tensor(u1, device="cuda")).cpu().numpy().astype(np.complex128)
        gu1, gd1 = gpu_adjoint(plan, u1, gu2)
    lhs, rhs = np.vdot(gu2.astype(np.complex128), fwd), np.vdot(gu1.astype(np.complex128), u1)
    assert abs(lhs - rhs) <= 1e-5 * np.linalg.norm(gu2) * np.linalg.norm(fwd), (lhs, rhs)
    cut = 3.0 * 10.0 ** (-(width - 1))
    assert rel_l2(gu1, ref_u1) < max(cut, 1e-5)
    assert rel_l2(gd1, ref_d1) < max(10 * cut, 1e-4)
