"""A chained launch that the runtime refuses gives its error to the caller and
leaves none behind for the next check of an unrelated launch (host only: the
launch asks for more threads than a block may have, or there is no device)."""
import os
import subprocess

from paper_1605_05320_gb300 import build as B

SRC = r"""
#include <stdio.h>
#include "chain.cuh"
__global__ void kernel(int *p) { swadj::chain_begin(); if (p) *p = 1; }
int main() {
    cudaGetLastError();
    const cudaError_t e =
        swadj::launch_chained(kernel, dim3(1), dim3(2048), 0, 0, (int *)nullptr);
    printf("%d %d\n", (int)e, (int)cudaGetLastError());
    return 0;
}
"""


def test_refused_launch_leaves_no_error_behind(tmp_path):
    src, exe = tmp_path / "launch.cu", str(tmp_path / "launch")
    src.write_text(SRC)
    subprocess.run([B._nvcc()] + B.NVCC_FLAGS + [str(src), "-o", exe], check=True,
                   capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    returned, left = (int(x) for x in r.stdout.split())
    assert returned != 0 and left == 0
