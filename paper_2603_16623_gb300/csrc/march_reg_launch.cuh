// march_reg_launch.cuh -- launch template of the register marches, shared by
// the translation units that instantiate them (AB2 in march_reg_ab2.cu, RK4
// in march_reg_rk4.cu, compiled in parallel).
#pragma once
#include "march.h"
#include "march_reg.cuh"

namespace gbwake {

template <class P>
inline cudaError_t launch_reg(void (*kern)(const WakeDev<P>*, const int32_t*, int32_t, int32_t),
                              const WakeDev<P>* d_wakes, const int32_t* d_order, int32_t n_wakes, int32_t max_slices,
                              int32_t mode, int32_t threads, int32_t cl, size_t smem, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cudaGetLastError(), e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_wakes * cl), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, d_wakes, d_order, max_slices, mode);
    if (e != cudaSuccess) return cudaGetLastError(), e;
    return cudaGetLastError();
}

}  // namespace gbwake
