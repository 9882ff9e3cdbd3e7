"""The prefactor's phase on the spreads that promise an accurate sine and cosine:
wrapping and folding maps of every width, widths 15 and 16, and maps of more
samples per kernel width than the lanes of a tile could hold apart.

A single sample's transform, divided by its exact value and averaged over the
destination's pairs of opposite points, is the sample's prefactor divided by its
own: errors of the position and of the (real) taps cancel in the pairs, the FFT's
rounding averages out.  The FP32 phase (a_x + a_y) q is formed here as the
library documents it, so that what is left is the rounding of the tables (2.4e-8
rms for both), of their product (2.4e-8), of sine and cosine (2e-8) and of the last
product (2.4e-8): 4.7e-8 rms over the samples.  Asked for: 7e-8.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import FresnelPlan  # noqa: E402

pytestmark = pytest.mark.gpu

LAM, Z0, M = 633e-9, 0.06, 64

# n1, p1, fine cells per sample, width, deterministic, heights: random (the map
# folds) or one value (it is monotone)
CASES = {
    "wrapping_w4": (512, 8e-6, 0.3, 4, False, "smooth"),
    "wrapping_w7": (512, 8e-6, 0.3, 7, False, "smooth"),
    "wrapping_w9": (512, 8e-6, 0.3, 9, False, "smooth"),
    "wrapping_w12": (512, 8e-6, 0.3, 12, False, "smooth"),
    "wrapping_w16": (512, 8e-6, 0.3, 16, False, "smooth"),
    "folding_w7": (512, 8e-6, 0.1, 7, False, "random"),
    "folding_w12": (512, 8e-6, 0.1, 12, False, "random"),
    "w15": (96, 42e-6, 1.03, 15, False, "flat"),
    "w16": (96, 42e-6, 1.03, 16, False, "flat"),
    "w16_close": (256, 16e-6, 0.4, 16, False, "flat"),
    "dense_w8": (512, 8e-6, 0.1, 8, False, "flat"),
    "dense_w12": (512, 8e-6, 0.1, 12, False, "flat"),
    "dense_w7_repeatable": (512, 8e-6, 0.1, 7, True, "flat"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_prefactor_phase(name):
    n, p1, alpha, width, det, heights = CASES[name]
    rng = np.random.default_rng(len(name))
    p2 = alpha * LAM * Z0 / (p1 * 2 * M)
    g = W.geometry(n, n, p1, p1, M, M, p2, p2, LAM, Z0)
    d1 = np.full((n, n), 2.9e-4)
    if heights == "random":
        d1 = rng.uniform(1e-4, 6e-4, (n, n))
    elif heights == "smooth":
        d1 = 1e-4 + W.surface_smooth_random(g, rng, 20.0, 2e-4)
    x1 = (np.arange(n) - n // 2) * p1
    a = (x1 * x1 / (LAM * Z0)).astype(np.float32)
    x2 = (np.arange(M) - M // 2) * p2
    outer = np.exp(1j * np.pi * ((2 * Z0 / LAM) % 2.0)) / 1j
    chirp = np.exp(1j * np.pi * x2 * x2 / (LAM * Z0))
    errs = []
    with FresnelPlan(g, d1, kernel_width=width, deterministic=det) as plan:
        for _ in range(96):
            ix, iy = (int(v) for v in rng.integers(0, n, 2))
            u = torch.zeros((n, n), dtype=torch.complex64, device="cuda")
            u[iy, ix] = 1.0
            got = plan.execute(u).cpu().numpy().astype(np.complex128)
            h = d1[iy, ix]
            q = np.float32(h) / np.float32(Z0 - h)
            ph = float(np.float32(a[ix] + a[iy]) * q)
            c = np.exp(1j * np.pi * ((x1[ix] ** 2 + x1[iy] ** 2) / (LAM * Z0) % 2.0 + ph))
            r0 = Z0 - h
            ref = (np.exp(-2j * np.pi * x2 * x1[iy] / (LAM * r0)) * chirp)[:, None] * \
                  (np.exp(-2j * np.pi * x2 * x1[ix] / (LAM * r0)) * chirp)[None, :] * (outer * c)
            # (without -M/2, which has no +M/2: real taps' errors cancel in pairs)
            errs.append(np.angle(np.vdot(ref[1:, 1:], got[1:, 1:])))
    rms = float(np.sqrt(np.mean(np.square(errs))))
    print(name, rms)
    assert rms < 7e-8, (name, rms, float(np.max(np.abs(errs))))
