// march_reg_ions.cu -- instantiations of the two-species march with rings in registers.
#include "march_reg_ions.cuh"

#include "march_reg_launch.cuh"

namespace gbwake {

template <class P>
cudaError_t launch_march_reg_ions(const WakeDev<P>* d_wakes, const int32_t* d_order, int32_t n_wakes,
                                  int32_t max_slices, int32_t mode, int32_t threads, int32_t k_rings, int32_t cl,
                                  int32_t n_max, cudaStream_t st) {
    const size_t smem = reg_smem_bytes<typename P::R>(n_max, 1);
    auto kern = k_rings == 1 ? march_ions_reg_kernel<P, 1> : march_ions_reg_kernel<P, 2>;
    return launch_reg(kern, d_wakes, d_order, n_wakes, max_slices, mode, threads, cl, smem, st);
}

template cudaError_t launch_march_reg_ions<PrecF64>(const WakeDev<PrecF64>*, const int32_t*, int32_t, int32_t, int32_t,
                                                    int32_t, int32_t, int32_t, int32_t, cudaStream_t);
template cudaError_t launch_march_reg_ions<PrecMixed>(const WakeDev<PrecMixed>*, const int32_t*, int32_t, int32_t,
                                                      int32_t, int32_t, int32_t, int32_t, int32_t, cudaStream_t);

}  // namespace gbwake
