// march_f64.cu -- launcher of the double-precision on-chip march, in a
// translation unit of its own so that it compiles in parallel.
#include "march_f64.cuh"
#include "march.h"

namespace gbwake {

template <int K>
static cudaError_t launch_f64_k(const WakeDev<PrecF64>* d_wakes, const int32_t* d_order, int32_t n_wakes,
                                int32_t max_slices, int32_t mode, int32_t threads, int32_t cl, int32_t n_max,
                                cudaStream_t st) {
    const size_t smem = f64_smem_bytes(n_max);
    cudaError_t e =
        cudaFuncSetAttribute(march_f64_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cudaGetLastError(), e;
    if (cl > 8) {
        e = cudaFuncSetAttribute(march_f64_kernel<K>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return cudaGetLastError(), e;
    }
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
    e = cudaLaunchKernelEx(&cfg, march_f64_kernel<K>, d_wakes, d_order, max_slices, mode);
    if (e != cudaSuccess) return cudaGetLastError(), e;
    return cudaGetLastError();
}

// Blocks of 128 threads: one warp per FP64 pipe of an SM (a warp's FP64
// instruction holds its sub-partition's pipe for 64 cycles, whatever else is
// in flight), so a second warp there only adds its share of the scans.
// Rings per thread: 1 up to 512 rings, 2 up to 4096, 4 beyond; measured on
// one wake alone (us per slice; 16 blocks at most): 500 rings 22.2 on 4 x 1,
// 26.2 on 2 x 2; 2000 rings 28.9 on 8 x 2, 26.6 on 16 x 1, 40.4 on 4 x 4;
// 4000 rings 32.0 on 16 x 2, 44.1 on 8 x 4; 8000 rings 52.0 on 16 x 4.  More
// rings per thread share a warp's scans between them, which is what counts
// when wakes fill the GPU (152 wakes of 2000 rings: 8 x 2 179, 16 x 1 212,
// 2 x 4 on 256 threads 114 us per slice): the middle one is taken, since a
// wake's shape is fixed before its batch is known.
F64Shape f64_shape(int32_t n) {
    constexpr int32_t kThreads = 128;
    F64Shape f;
    f.k = n <= 512 ? 1 : n <= 4096 ? 2 : 4;
    f.cl = (n + kThreads * f.k - 1) / (kThreads * f.k);
    const int32_t per = (n + f.cl - 1) / f.cl;
    f.threads = ((per + f.k - 1) / f.k + 31) / 32 * 32;
    while (f.cl > 1 && (int64_t)f.threads * f.k * (f.cl - 1) >= n) --f.cl;  // (no block without a ring)
    return f;
}

cudaError_t launch_march_f64(const WakeDev<PrecF64>* d_wakes, const int32_t* d_order, int32_t n_wakes,
                             int32_t max_slices, int32_t mode, int32_t threads, int32_t k_rings, int32_t cl,
                             int32_t n_max, cudaStream_t st) {
    if (k_rings == 1)
        return launch_f64_k<1>(d_wakes, d_order, n_wakes, max_slices, mode, threads, cl, n_max, st);
    if (k_rings == 2)
        return launch_f64_k<2>(d_wakes, d_order, n_wakes, max_slices, mode, threads, cl, n_max, st);
    return launch_f64_k<4>(d_wakes, d_order, n_wakes, max_slices, mode, threads, cl, n_max, st);
}

}  // namespace gbwake
