// launch.cuh -- launch of a kernel behind the kernel before it on its stream.
#pragma once

#include <cuda_runtime.h>

namespace scale {

// Launch `kern` so that its CTAs may become resident before the kernel ahead of
// it on `st` has completed (it waits with scale_ptx::pdl_wait): the launch and
// the first instructions hide behind that kernel's end. Back to back, empty
// kernels take 1.4 us each this way and 2.1 us otherwise. `cluster` > 1: CTAs of
// a cluster along x.
template <typename... Params, typename... Args>
cudaError_t launch_after(cudaStream_t st, dim3 grid, unsigned threads, size_t smem, unsigned cluster,
                         void (*kern)(Params...), const Args&... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2]{};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
    if (e != cudaSuccess) cudaGetLastError();  // reported by the return value
    return e;
}

}  // namespace scale
