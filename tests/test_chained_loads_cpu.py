"""Kernels launched with programmatic serialisation may run while their inputs are
still written: they must not read them through the non-coherent path.  In the
sources: __ldg, and const __restrict__ parameters of such kernels (which the
compiler turns into the same loads), are for tables that were complete before a
call of the host's returned.
"""
from __future__ import annotations

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1203_3583_gb300", "csrc")
# q (asfd_plan_update_d1 waits for it), twiddles, deconvolution (learned_refresh ends
# the chain after it writes them), the line plan's and the item tiles' tables
TABLES = {"q", "tw", "cx", "cy", "e", "bi", "bf", "C", "xbox", "ybox", "xmap", "ymap"}


def sources():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(f).read())
        yield os.path.basename(f), text


def test_ldg_reads_tables_only():
    seen = 0
    for name, text in sources():
        for m in re.finditer(r"__ldg\(\s*(.{0,60})", text, flags=re.S):
            seen += 1
            op = re.match(r"&(?:\w+\.)?(\w+)\s*\[", m.group(1))
            assert op and op.group(1) in TABLES, (name, m.group(0))
    assert seen > 5


def test_chained_kernels_have_no_restricted_inputs():
    text = "\n".join(t for _, t in sources())
    chained = set()
    for m in re.finditer(r"launch_chained\(([^;]*?);", text, flags=re.S):
        chained |= set(re.findall(r"\b(\w+_kernel)\b", m.group(1)))
    chained.add("spread_block_kernel")  # through a table of instances
    assert {"fft_rows_kernel", "loss_kernel", "table_grad_kernel", "direct_sum_kernel"} <= chained
    for k in sorted(chained):
        m = re.search(r"__global__[^;{]*?\b%s\(([^)]*)\)" % k, text, flags=re.S)
        assert m, k
        for p in m.group(1).split(","):
            r = re.search(r"\bconst\b.*__restrict__\s+(\w+)", p, flags=re.S)
            assert not r or r.group(1) in TABLES, (k, p)
