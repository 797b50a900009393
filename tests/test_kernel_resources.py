"""The batched cell kernels keep their lines in registers.

A batch's kernels carry the bodies of the single-problem kernels, whose n values
per line live in registers; a kernel that holds too much at once (every
degree's body, say) moves them to local memory, through the data pipe that
bounds these passes.  The compiler's own report (ptxas -v) names the stack
bytes of every kernel: none for the DG passes.
"""
import os
import re
import subprocess

import pytest

from paper_1910_01900_gb300 import build


@pytest.mark.parametrize("source,kernels", [("batch.cu", ("dg_batched_kernel", "dg_box_batched_kernel"))])
def test_batched_cell_kernels_use_no_local_memory(source, kernels, tmp_path):
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    cmd = [nvcc] + build.ARCH + build.COMMON + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, source),
                                                "-o", str(tmp_path / "k.o")]
    out = subprocess.run(cmd, capture_output=True, text=True, check=True).stderr
    stack = re.findall(r"Function properties for (\S+)\s+(\d+) bytes stack frame", out)
    for k in kernels:
        mine = [(name, int(b)) for name, b in stack if re.search(r"\d%sI" % k, name)]
        assert mine, k
        assert [x for x in mine if x[1]] == []
