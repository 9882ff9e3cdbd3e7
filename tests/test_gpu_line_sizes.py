"""The 1D transform where its launch changes: one block up to 1024 samples and
two per fine cell, a spread kernel of its own above; lines of 64 to 16384 fine cells (4 to 1024
transform threads); and a line that holds nothing over from call to call.
Tolerance as in test_gpu_line: the width's truncation or 5e-6.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import line as oline  # noqa: E402
from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import LinePlan  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m2,width", [(1, 32, 7), (33, 64, 16), (128, 32, 7), (129, 32, 5),
                                        (1024, 512, 7), (1025, 512, 2), (20000, 4096, 9), (700, 8192, 6)])
def test_line_sizes(n, m2, width):
    rng = np.random.default_rng(n + m2)
    x1 = rng.uniform(-1.5e-3, 1.5e-3, n)
    d1 = rng.uniform(-2e-5, 2e-5, n)
    w = rng.uniform(0.5, 1.5, n) * 3e-3 / n
    line = W.line_geometry(m2=m2, p2=4e-6, lam=532e-9, z0=0.4)
    us = [(rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64) for _ in range(2)]
    with LinePlan(line, x1, d1, w, kernel_width=width) as p:
        got = [p.execute(torch.as_tensor(u, device="cuda")).cpu().numpy() for u in us + us[:1]]
        zero = p.execute(torch.zeros(n, dtype=torch.complex64, device="cuda"))
        assert torch.count_nonzero(zero).item() == 0
    for g, u in zip(got, us + us[:1]):
        ref = oline.line(line, x1, d1, w, u.astype(np.complex128), 7)
        err = np.linalg.norm(g - ref) / np.linalg.norm(ref)
        assert err < max(5e-6, 3.0 * 10.0 ** (-(width - 1))), (n, m2, width, err)
