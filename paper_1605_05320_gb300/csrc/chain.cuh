// chain.cuh -- chained launches of the step kernels.
//
// A step sequence is one kernel after another on one stream, each a few to
// tens of microseconds.  Launched plainly, the next kernel starts after the
// last block of the one before has left and its writes are flushed, and the
// GPU idles meanwhile.  Chained kernels (programmatic stream serialisation)
// are set up while the kernel before still runs: their blocks take the SMs
// as its blocks leave and wait in chain_begin() until it has completed and
// its writes are visible.  Every thread of a chained kernel calls
// chain_begin() before it reads or writes global memory.
// Measured, us per step, plain / chained: FP32 forward 64^2 12.3 / 10.3, 512^2
// at rest outside the source 15.0 / 12.7, 2048^2 37.3 / 35.0 and with waves
// everywhere 71.8 / 70.0; FP32 adjoint 512^2 8.2 / 5.8, 2048^2 early 19.9 / 17.5
// and late 36.4 / 34.4.  The blocks of a chained kernel take the slots that become
// free first, so that some SMs can hold more than their share while others idle.
// The FP64 sweeps, which the FP64 units bound, are not chained for that (adjoint,
// 512^2 late: 103 plain, 140 chained; forward, whose units come from a counter once a
// block is placed, 256 x 200: 101 and 117), and kernels whose blocks take one share
// of the work each are chained by their number (launch_spread).  The FP64 1D step, in
// blocks of one warp, is chained at all sizes (2000 cells 12.9 and 11.3, 100000 34.2
// and 32.2).
#pragma once
#include <cuda_runtime.h>

namespace swadj {

__device__ __forceinline__ void chain_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t st, const A &...args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();   // returned here, not left for a later check
    return e;
}

}  // namespace swadj
