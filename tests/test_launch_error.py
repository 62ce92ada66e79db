"""A chained launch that the runtime refuses gives its error to the caller and
leaves none behind for the next check of an unrelated launch (host only: the
launcher compiled against a fake of the CUDA calls it makes)."""
import subprocess

from paper_1605_05320_gb300 import build as B

FAKE = r"""
#pragma once
#include <stddef.h>
#define __device__
#define __forceinline__ inline
struct dim3 { unsigned x, y, z; dim3(unsigned a = 1) : x(a), y(1), z(1) {} };
typedef int cudaError_t;
typedef void *cudaStream_t;
enum { cudaSuccess = 0, cudaLaunchAttributeProgrammaticStreamSerialization = 6 };
struct cudaLaunchAttribute {
    int id;
    struct { int programmaticStreamSerializationAllowed; } val;
};
struct cudaLaunchConfig_t {
    dim3 gridDim, blockDim;
    size_t dynamicSmemBytes;
    cudaStream_t stream;
    cudaLaunchAttribute *attrs;
    unsigned numAttrs;
};
inline cudaError_t &last_error() { static cudaError_t e = cudaSuccess; return e; }
inline cudaError_t cudaGetLastError() {
    const cudaError_t e = last_error();
    last_error() = cudaSuccess;
    return e;
}
template <typename... P, typename... A>
cudaError_t cudaLaunchKernelEx(const cudaLaunchConfig_t *c, void (*)(P...), A &&...) {
    return c->blockDim.x > 1024 ? last_error() = 9 : cudaSuccess;
}
"""

MAIN = r"""
#include <stdio.h>
#include "chain.cuh"
void kernel(int *) {}
int main() {
    int *p = nullptr;
    const cudaError_t e = swadj::launch_chained(kernel, dim3(1), dim3(2048), 0, 0, p);
    printf("%d %d ", e, cudaGetLastError());
    last_error() = 3;   // an error of someone else's is not taken away
    const cudaError_t f = swadj::launch_chained(kernel, dim3(1), dim3(128), 0, 0, p);
    printf("%d %d\n", f, cudaGetLastError());
    return 0;
}
"""


def test_refused_launch_leaves_no_error_behind(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    (tmp_path / "main.cc").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run(["g++", "-std=c++17", f"-I{tmp_path}", f"-I{B.CSRC}",
                    str(tmp_path / "main.cc"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.stdout.split() == ["9", "0", "0", "3"]
