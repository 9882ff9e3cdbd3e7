"""Eq. 2's distance at ranges of many wavelengths: r enters the phase as
2 r / lambda half-turns, 2.2e7 of them at 5 m and 450 nm, so it has to be as good
as an FP64 square root.

Reference: r - z0 = (dx^2 + dy^2 - d1 (2 z0 - d1)) / (r + z0) in FP64 (good to
1e-16 of a small number), with the constant phase of z0 apart.
Tolerance: per term of a sum, relative to its size and rms, 2.4e-8 sine and
cosine, 2.4e-8 products, 2e-8 amplitude, 2e-8 the FP64 phase of 2.2e7 half-turns
(ulp of r times 2 pi / lambda): 4.5e-8; the output's rounding 3e-8; so below
1e-7 with every part at twice its rms, and 2e-7 is asked for.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import direct_sum  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-14, 1e16])
@pytest.mark.parametrize("z0,lam", [(0.15, 532e-9), (1.0, 450e-9), (5.0, 450e-9), (40.0, 450e-9)])
def test_distance_is_exact(z0, lam, scale):
    """scale: the geometry in other units; r^2 then leaves FP32's range."""
    rng = np.random.default_rng(int(z0 * 10) if scale == 1.0 else 1)
    n, m = 96, 64
    z0, lam, p1, p2 = z0 * scale, lam * scale, 10e-6 * scale, 20e-6 * scale
    g = W.geometry(n, n, p1, p1, m, m, p2, p2, lam, z0)
    d1 = rng.uniform(-2e-3, 2e-3, (n, n)) * scale
    u1 = W.field_random_amp_phase(g, rng)
    mx, my = (rng.integers(0, m, 24).astype(np.int32) for _ in range(2))
    got = direct_sum(g, d1, torch.as_tensor(u1, device="cuda"), 2, (mx, my)).cpu().numpy()
    x1 = (np.arange(n) - n // 2) * g["p1x"]
    dx = ((mx - m // 2) * g["p2x"])[:, None, None] - x1[None, None, :]
    dy = ((my - m // 2) * g["p2y"])[:, None, None] - x1[None, :, None]
    rho2 = dx * dx + dy * dy
    r = np.sqrt(rho2 + (z0 - d1) ** 2)
    turns = ((rho2 - d1 * (2 * z0 - d1)) / (r + z0) + d1) / lam  # exp(ik(d1 + r - z0))
    turns -= np.rint(turns)
    ref = (u1.astype(np.complex128) * np.exp(2j * np.pi * turns) / r ** 2).sum((1, 2))
    half = 2 * z0 / lam
    half -= 2 * np.rint(half / 2)
    ref = ref * np.exp(1j * np.pi * half) * g["p1x"] * g["p1y"] * z0 / (1j * lam)
    err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
    # (z0 / lambda in FP64 is one common phase)
    assert err < 2e-7 + 2 * np.pi * z0 / lam * 2.0 ** -53, (z0, err)
