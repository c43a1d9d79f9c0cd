"""Set-up tables reach the device on the stream of the kernels that read them (no GPU needed)."""

import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2103_10203_gb300", "csrc")


def test_no_upload_on_the_legacy_stream():
    """cudaMemcpy from pageable memory and cudaMemset may return while the device still works on them,
    on a stream that non-blocking streams do not wait for."""
    found = []
    for name in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"\bcudaMem(?:cpy|set)\((.*?);", src, re.S):
            if "cudaMemset" in m.group(0) or "HostToDevice" in m.group(1):
                found.append((name, src.count("\n", 0, m.start()) + 1))
    assert not found
