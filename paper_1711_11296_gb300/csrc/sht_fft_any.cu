// FP32 FFT kernels with the shape known at run time (regular grids and the
// rows of reduced grids).
#include "sht_fft_kernels.h"

namespace sht {

cudaError_t fft_any_init() { return upload_twiddles(); }

cudaError_t fft_any_forward(const FwdArgs<float>& A, bool strided, dim3 grid, size_t smem,
                            cudaStream_t s, Follow follow) {
    if (!strided) return fft_launch(fft_forward_kernel<float, -1, false>, A, grid, smem, s, follow);
    return fft_launch(fft_forward_kernel<float, -1, true>, A, grid, smem, s, follow);
}

cudaError_t fft_any_inverse(const InvArgs<float>& A, dim3 grid, size_t smem, cudaStream_t s, Follow follow) {
    return fft_launch(fft_inverse_kernel<float, -1>, A, grid, smem, s, follow);
}

cudaError_t fft_any_forward_ragged(const RaggedFwd<float>& R, dim3 grid, size_t smem,
                                   cudaStream_t s, Follow follow) {
    return fft_launch(fft_forward_ragged_kernel<float>, R, grid, smem, s, follow);
}

cudaError_t fft_any_inverse_ragged(const RaggedInv<float>& R, dim3 grid, size_t smem,
                                   cudaStream_t s, Follow follow) {
    return fft_launch(fft_inverse_ragged_kernel<float>, R, grid, smem, s, follow);
}

}  // namespace sht
