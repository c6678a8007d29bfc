// launch.h -- launches with programmatic stream serialization.
#pragma once
#include <cuda_runtime.h>

namespace ebit {

// Launch with programmatic stream serialization: the kernel is launched as
// the previous kernel's blocks exit, and waits (pdl_wait) for that kernel's
// completion before it touches global memory.  Counters that a
// launch appends to are cleared by an earlier kernel of the chain (in its
// zero arguments) instead of by memsets, which would break the overlap.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// The id of the capture that a stream's work is recorded into (0: it runs).  Work
// that a replay repeats must not lean on lists that were made outside its graph.
inline unsigned long long capture_id(cudaStream_t st) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamGetCaptureInfo(st, &status, &id) != cudaSuccess) cudaGetLastError();
    return status == cudaStreamCaptureStatusActive ? id : 0;
}

}  // namespace ebit
