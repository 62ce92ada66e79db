"""GPU test of the FP64 division and square root where the integer path ends:
the compiler's bits, the sign of a zero included, at both ends of the normal
numbers and for zeros, subnormals, infinities and NaN."""
import os
import subprocess

import pytest

from paper_1605_05320_gb300 import build as B

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_edges_of_division_and_root(tmp_path):
    exe = str(tmp_path / "ops64_edges_check")
    src = os.path.join(HERE, "native", "ops64_edges_check.cu")
    subprocess.run([B._nvcc(), "-fmad=false"] + B.NVCC_FLAGS + [src, "-o", exe], check=True,
                   capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
