"""The registers of the tensor-core backward stay registers.

The backward composite holds the destination of a tensor-memory load across a
pair's work and waits for the load after it.  Until that wait the register has
no value yet: a compiler that spilled it in between would store garbage."""
import os
import re
import subprocess

import pytest

from paper_2510_12174_gb300 import build as b


def test_tensor_core_backward_does_not_spill(tmp_path):
    try:
        nvcc = b._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    r = subprocess.run([nvcc, *b.NVCC_FLAGS, "-Xptxas", "-v", "-c",
                        os.path.join(b.CSRC, "render_bwd_tc.cu"), "-o", str(tmp_path / "k.o")],
                       capture_output=True, text=True, check=True)
    found = re.findall(r"Function properties for \S*render_bwd_tc_kernel\S*\n\s*(.*)", r.stderr)
    assert len(found) == 3  # 16, 32 and 64 logits
    for line in found:
        assert line.startswith("0 bytes stack frame, 0 bytes spill stores, 0 bytes spill loads")
