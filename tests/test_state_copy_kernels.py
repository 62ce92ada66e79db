"""The kernels that copy a state out keep their parameters out of local memory:
indexing an array of pointers in a kernel's parameters by a value known on the
device only gives every thread a copy of them (host only: the compiler's
report)."""
import os
import re
import subprocess

import pytest

from paper_1605_05320_gb300 import build as B


@pytest.mark.parametrize("source,kernel", [("api.cu", "state_out_kernel"),
                                           ("patches.cu", "patch_out_kernel")])
def test_no_stack_frame(tmp_path, source, kernel):
    r = subprocess.run([B._nvcc(), "-Xptxas=-v"] + B.NVCC_FLAGS +
                       ["-c", os.path.join(B.CSRC, source), "-o", str(tmp_path / "x.o")],
                       check=True, capture_output=True, text=True)
    out = r.stdout + r.stderr
    frames = re.findall(r"Compiling entry function '(\w*%s\w*)'.*?(\d+) bytes stack frame" % kernel,
                        out, re.S)
    assert frames and all(int(n) == 0 for _, n in frames), frames
