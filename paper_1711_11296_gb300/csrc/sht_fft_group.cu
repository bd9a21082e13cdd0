// Grouped FP32 FFT kernels: several plans' rows in one launch.
#include "sht_fft_kernels.h"

namespace sht {

cudaError_t fft_group_init() { return upload_twiddles(); }

cudaError_t fft_group_forward(const FwdGroup<float>& G, int ctas, size_t smem, cudaStream_t s,
                              Follow follow) {
    return fft_launch(fft_forward_group_kernel<float>, G, dim3(ctas), smem, s, follow);
}

cudaError_t fft_group_inverse(const InvGroup<float>& G, int ctas, size_t smem, cudaStream_t s,
                              Follow follow) {
    return fft_launch(fft_inverse_group_kernel<float>, G, dim3(ctas), smem, s, follow);
}

}  // namespace sht
