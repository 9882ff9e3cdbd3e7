"""The one-block transform of a line of 8192 fine cells, whose block has 512 threads
for up to 1024 samples.  Tolerance as in test_gpu_line (5e-6 at width 7)."""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import line as oline  # noqa: E402
from paper_1203_3583_gb300 import workloads as W  # noqa: E402
from paper_1203_3583_gb300.fresnel import LinePlan  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 512, 513, 1024, 1025])
def test_line_of_8192_cells(n):
    rng = np.random.default_rng(n)
    x1 = rng.uniform(-1.5e-3, 1.5e-3, n)
    d1 = rng.uniform(-2e-5, 2e-5, n)
    w = rng.uniform(0.5, 1.5, n) * 3e-3 / n
    line = W.line_geometry(m2=4096, p2=4e-6, lam=532e-9, z0=0.4)
    u = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)
    with LinePlan(line, x1, d1, w) as p:
        got = p.execute(torch.as_tensor(u, device="cuda")).cpu().numpy()
    ref = oline.line(line, x1, d1, w, u.astype(np.complex128), 7)
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) < 5e-6
