// Programmatic dependent launch of the kernels that follow one another closely (split, contraction, solve;
// proposal, accept; the surrogate's products). A kernel launched with launch_after may be resident before
// its predecessor in the stream has finished, so that its launch and prologue overlap the predecessor's
// end; it calls grid_wait() with every thread before it touches global memory, which returns when the
// predecessor has finished and its writes are visible. Each kernel of a chain waits before it can end, so
// waiting for the direct predecessor is waiting for all of them. What bounds such a chain is the gap between
// its launches, about 2 us each: 100 particles on 1/8 53 -> 49 us, a tempering update of 1000 particles on 1/32 (33
// such launches) 684 -> 620 us, a gradient pass of the surrogate (24) 343 -> 284 us.
// A successor comes in as the predecessor's blocks end, never earlier (griddepcontrol.launch_dependents): blocks
// that come in while some SMs are still taken are stacked on the others, and a solve is as slow as its fullest
// SM. With that trigger at the start of every kernel an FP64 tempering update of 1000 particles on 1/8 took 2069
// us (1020 without), of 450 on 1/16 2210 (1656), 300 particles on 1/32 47.5 (35.8), 4000 on 1/8 55.5 (50.6).
#pragma once

#include <cuda_runtime.h>

namespace mls2mc {

// every thread of a kernel launched with launch_after, before its first global access (returns at once
// in a kernel launched without the attribute)
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

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
