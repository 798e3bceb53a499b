// Launches that overlap a kernel's start with the end of the kernel before it in the stream.
//
// A kernel launched with chained = true may start once every block of the preceding kernel has
// called grid_release() or ended; it calls grid_wait() before its first access to memory another
// kernel may write or read, which returns when the preceding kernel has completed.  Kernels that
// call neither behave as ever on both sides.  What overlaps is the launch itself, block scheduling,
// barrier and tensor-memory set-up: some 2 us of a call (64 inputs x 128 channels x 512 4-bit samples,
// calls back to back: 10.5 -> 8.4 us; filterbank + X stage 375 -> 372; phasors + fused dump 152 -> 148).
// Only the packed-sample tensor-core kernels are chained.  Chained as well, the kernels before them
// (unpack, F stage, phasors) started under the previous call's X stage and slowed the pair: 375 ->
// 418 us for the filterbank chain, 408 -> 440 for a 400-input dump from planes; nor did the plane-fed
// kernel gain behind its unpack (408 -> 417).
#pragma once

#include <cuda_runtime.h>

namespace corr {

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// cluster: blocks per cluster along x (1: none).  Under stream capture the plain dependency is kept.
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kern)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, int cluster,
                          bool chained, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    int n = 0;
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = (unsigned)cluster;
        at[n].val.clusterDim.y = at[n].val.clusterDim.z = 1;
        ++n;
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (chained && cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = at;
    cfg.numAttrs = (unsigned)n;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

}  // namespace corr
