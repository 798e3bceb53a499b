// Kernel launches with cluster dimensions.
#pragma once

#include <cuda_runtime.h>

namespace corr {

// cluster: blocks per cluster along x (1: none).
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kern)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, int cluster,
                          bool /*chained*/, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

}  // namespace corr
