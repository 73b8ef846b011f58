// direct_launch.cuh -- the cluster launch of direct.cuh, included by the files
// that compile one shape's kernel each.
#pragma once

#include "direct.cuh"

namespace lms {
namespace direct {

// An error (not launched) also where the device cannot hold the cluster: the
// caller then takes the path of many kernels.
template <class SH>
cudaError_t launch_cluster(const DirectArgs &a, size_t smem, cudaStream_t st)
{
    auto kern = SH::kernel();
    const int C = a.shape.C;
    cudaError_t e = allow_smem(kern, smem);
    if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(SH::T);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (!cluster_fits(reinterpret_cast<const void *>(kern), cfg)) return cudaErrorLaunchOutOfResources;
    StageTimer _t(STAGE_DIRECT, st);
    return cudaLaunchKernelEx(&cfg, kern, a);
}

}  // namespace direct
}  // namespace lms
