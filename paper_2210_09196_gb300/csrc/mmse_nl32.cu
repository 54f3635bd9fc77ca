// MMSE detection kernels of the 32-layer class (kernel in mmse_impl.cuh).
#include "mmse_impl.cuh"

namespace pusch {

cudaError_t mmse_launch_class32(const mmse_detail::MmseArgs &a, long long total_sc, const float2 *H,
                                const float2 *beam, const float2 *ls, const float *sigma2, float2 *xhat,
                                uint8_t *bits, uint32_t *status, cudaStream_t st) {
    return mmse_detail::launch_nd<32>(a, total_sc, H, beam, ls, sigma2, xhat, bits, status, st);
}

}  // namespace pusch
