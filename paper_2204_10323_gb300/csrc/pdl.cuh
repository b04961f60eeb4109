// pdl.cuh -- programmatic dependent launch: a kernel launched through launch_pdl may be put on the
// SMs while the one before it in the stream still runs, and waits there (pdl_wait, before its first
// access to global memory) until that one has completed and its writes are visible.  The chain of
// small dependent kernels that a step loop is then loses its launch gaps (a launch after a launch otherwise
// costs one to three microseconds, in steps of two).  pdl_launch, after the wait, lets the next one come.
#pragma once

#include <cuda_runtime.h>

namespace flood {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Every kernel launched so calls pdl_wait in all its threads first.  Captured launches keep plain edges.
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(st, &capture);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = capture == cudaStreamCaptureStatusNone ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace flood
