"""Host memory that a copy from the device fills is read only after a wait: a copy
to pageable memory may return before it has ended.  In the sources of plan creation
and update: after copies to the host the next statement waits for the stream."""
from __future__ import annotations

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1203_3583_gb300", "csrc")


@pytest.mark.parametrize("name,copies", [("plan.cu", 4), ("spread_item.cu", 2)])
def test_copies_to_the_host_are_waited_for(name, copies):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    found = list(re.finditer(r"cudaMemcpyAsync\([^;]*cudaMemcpyDeviceToHost[^;]*;", text))
    assert len(found) == copies
    for m in found:
        rest = re.sub(r"^(\s*ASFD_CUDA\(cudaMemcpyAsync\([^;]*;)+", "", text[m.end():])
        assert re.match(r"\s*ASFD_CUDA\(cudaStreamSynchronize\(st\)\);", rest), m.group(0)
