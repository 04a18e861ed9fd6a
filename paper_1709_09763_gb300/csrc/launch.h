// Programmatic dependent launch of the kernels that follow one another closely (split, contraction, solve;
// proposal, accept; the surrogate's products). A kernel launched with launch_after may be resident before
// its predecessor in the stream has finished, so that its launch and prologue overlap the predecessor's
// end; it calls grid_wait() with every thread before it touches global memory, which returns when the
// predecessor has finished and its writes are visible. grid_release() lets the next such kernel come in
// once every block of this one has called it or ended. Each kernel of a chain waits before it can end, so
// waiting for the direct predecessor is waiting for all of them. What bounds such a chain is the gap between
// its launches: 100 particles on 1/8 53 -> 49 us, 4000 on 1/32 190 -> 183 us, a tempering update of 1000
// particles (33 such launches) 684 -> 626 us, a gradient pass of the surrogate (24) 343 -> 285 us.
#pragma once

#include <cuda_runtime.h>

namespace mls2mc {

// every thread of a kernel launched with launch_after, before its first global access (returns at once
// in a kernel launched without the attribute)
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Plain launches while the stream is captured: a graph keeps full dependencies (and in-place updates).
inline bool may_overlap(cudaStream_t st) {
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &s) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return s == cudaStreamCaptureStatusNone;
}
inline void overlap_attr(cudaLaunchAttribute& a) {
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
}

template <typename... Params, typename... Args>
cudaError_t launch_after(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    overlap_attr(attr);
    cfg.attrs = &attr;
    cfg.numAttrs = may_overlap(st) ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

}  // namespace mls2mc
