// FP32 FFT kernels with the shape known at run time (regular grids and the
// rows of reduced grids).  Regular grids whose radices are small run a
// kernel that holds no others.
#include "sht_fft_kernels.h"

namespace sht {

namespace {
bool small_shape(const FftShape& sh) {
    for (int q = 0; q < sh.npass; ++q)
        if (sh.radix[q] > kSmallRadix) return false;
    return true;
}
}  // namespace

cudaError_t fft_any_init() { return upload_twiddles(); }

cudaError_t fft_any_forward(const FwdArgs<float>& A, bool strided, dim3 grid, size_t smem,
                            cudaStream_t s, Follow follow) {
    if (small_shape(A.shape)) {
        if (!strided)
            return fft_launch(fft_forward_kernel<float, -3, false>, A, grid, smem, s, follow);
        return fft_launch(fft_forward_kernel<float, -3, true>, A, grid, smem, s, follow);
    }
    if (!strided) return fft_launch(fft_forward_kernel<float, -1, false>, A, grid, smem, s, follow);
    return fft_launch(fft_forward_kernel<float, -1, true>, A, grid, smem, s, follow);
}

cudaError_t fft_any_inverse(const InvArgs<float>& A, dim3 grid, size_t smem, cudaStream_t s,
                            Follow follow) {
    if (small_shape(A.shape))
        return fft_launch(fft_inverse_kernel<float, -3>, A, grid, smem, s, follow);
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
