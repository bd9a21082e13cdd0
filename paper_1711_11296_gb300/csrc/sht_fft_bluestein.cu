// FFT kernels of reduced-grid rows whose half-length has a prime factor above
// 5 (Bluestein's method), FP32 and FP64.
#include "sht_fft_kernels.h"

namespace sht {

cudaError_t fft_bluestein_init() { return upload_twiddles(); }

cudaError_t fft_bluestein_forward(const RaggedFwd<float>& R, dim3 grid, size_t smem,
                                  cudaStream_t s, Follow follow) {
    return fft_launch(fft_forward_bluestein_kernel<float>, R, grid, smem, s, follow);
}

cudaError_t fft_bluestein_forward(const RaggedFwd<double>& R, dim3 grid, size_t smem,
                                  cudaStream_t s, Follow follow) {
    return fft_launch(fft_forward_bluestein_kernel<double>, R, grid, smem, s, follow);
}

cudaError_t fft_bluestein_inverse(const RaggedInv<float>& R, dim3 grid, size_t smem,
                                  cudaStream_t s, Follow follow) {
    return fft_launch(fft_inverse_bluestein_kernel<float>, R, grid, smem, s, follow);
}

cudaError_t fft_bluestein_inverse(const RaggedInv<double>& R, dim3 grid, size_t smem,
                                  cudaStream_t s, Follow follow) {
    return fft_launch(fft_inverse_bluestein_kernel<double>, R, grid, smem, s, follow);
}

}  // namespace sht
