"""The line transform keeps its values in registers at every length: no kernel of
line.cu spills, by the compiler's own report."""
from __future__ import annotations

import os
import re
import subprocess

from paper_1203_3583_gb300 import _build


def test_no_spills(tmp_path):
    src = os.path.join(_build.CSRC, "line.cu")
    cmd = [_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-Xptxas", "-v", "-c", src, "-o",
           str(tmp_path / "line.o")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    spills = dict(zip(re.findall(r"entry function '(\w+)'", r.stderr),
                      re.findall(r"(\d+) bytes spill stores", r.stderr)))
    assert sum("line_transform_kernel" in k for k in spills) == 18  # 9 lengths, with and without a spread
    assert {k: v for k, v in spills.items() if v != "0"} == {}
