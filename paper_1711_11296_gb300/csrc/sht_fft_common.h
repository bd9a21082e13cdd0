// Pieces shared by the FP32 FFT kernels (sht_fft.cu) and the fixed-point FFT
// kernels of the FP64 path (sht_fft64.cu): launch arguments, the padded row
// layout, asynchronous copies and index walks.
#pragma once

#include <type_traits>

#include "sht_internal.h"

namespace sht {

constexpr int kFftThreads = 256;   // threads per FFT CTA (two CTAs per SM)

// The plan's factorisation as a compile-time constant.
template <int L, bool FP64> struct FacOf {
    static constexpr FftShape v = fft_factor(L, FP64);
};

// Asynchronous global -> shared copy of one element (cp.async, no register
// staging, so all of a thread's copies are in flight at once).
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES)
                     : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

template <typename T>
__device__ __forceinline__ int ph(int pos) {
    return pos + (pos >> PadShift<T>::value);
}

// Digit-reversed position of frequency k.
template <typename T, int L>
__device__ __forceinline__ int rev_fixed(int k) {
    constexpr FftShape F = FacOf<L, sizeof(T) == 8>::v;
    int pos = 0;
#pragma unroll
    for (int q = 0; q < F.npass; ++q) {
        pos += (k % F.radix[q]) * F.span[q];
        k /= F.radix[q];
    }
    return pos;
}

template <typename T>
struct FwdArgs {
    using V = typename Vec2<T>::type;
    const T* grid;
    RowSource src;
    V* work;
    const V* twp;      // per-pass twiddle tables
    const V* twpost;
    const int* rev;
    const double* rowscale;
    double mscale0, mscale1;
    unsigned* colmax;   // FP16 split plans: max |output| per real column (float bits)
    const long long* rowoff;   // reduced grid: first point of each row (null: regular)
    const int* jh_list;        // latitude pair of each CTA row (null: blockIdx.y)
    const V* shiftph;          // rows shifted by half a spacing: e^{-i pi m / I_j} (else null)
    const V* chirp;            // Bluestein rows: e^{-i pi n^2 / L}
    const V* dft;              // Bluestein rows: DFT of the conjugate chirp / L2
    int F, J, Jh, L, LP, N, G;
    int follow;                // see Follow
    FftShape shape;
};

template <typename T>
struct InvArgs {
    using V = typename Vec2<T>::type;
    const V* work;
    T* grid;
    const V* twp;
    const V* twpost;
    const int* rev;
    const double* rowscale;
    double mfactor1;
    const long long* rowoff;   // reduced grid: first point of each row (null: regular)
    long long fstride;         // reduced grid: points per field
    const int* jh_list;        // latitude pair of each CTA row (null: blockIdx.y)
    int accumulate;            // 1: grid += rows (prolongation of a correction);
                               // 2: products (Sec. 4.2): with w the synthesised
                               // value, grid holds u and becomes u v, grid2
                               // holds v and becomes u v w
    T* grid2;                  // second grid of the products (else null)
    const V* shiftph;          // rows shifted by half a spacing: e^{-i pi m / I_j} (else null)
    const V* chirp;            // Bluestein rows: e^{-i pi n^2 / L}
    const V* dft;              // Bluestein rows: DFT of the conjugate chirp / L2
    int F, J, Jh, I, L, LP, N, G;
    int follow;                // see Follow
    FftShape shape;
};

// Copy the per-pass twiddle tables into shared memory asynchronously, so
// that they are in flight together with the CTA's data copies (one wait).
template <typename V>
__device__ __forceinline__ void load_twiddles_async(V* dst, const V* src, int n) {
    for (int e = threadIdx.x; e < n; e += kFftThreads) cp_async<sizeof(V)>(dst + e, src + e);
}

// The same by plain loads and stores (measured faster ahead of the inverse
// kernel's gathered copies).
template <typename V>
__device__ __forceinline__ void load_twiddles(V* dst, const V* src, int n) {
    for (int e = threadIdx.x; e < n; e += kFftThreads) dst[e] = src[e];
}

template <typename T, int LT>
__device__ __forceinline__ int rev_of(int k, const int* rev) {
    if constexpr (LT > 0)
        return rev_fixed<T, LT>(k);
    else if constexpr (LT == -2)
        return k;   // Bluestein rows end in natural order
    else
        return rev[k];
}

// Padded pitch of a row of n complex values (fft_row_pitch on the device).
template <typename T>
__device__ __forceinline__ int row_pitch(int n) {
    return n + (n >> PadShift<T>::value) + 1;
}

// How an FFT launch follows the kernel before it in the stream.
// The launches of one reduced-grid FFT (a class per row length, the run-time
// shapes, Bluestein rows) work on different rows and may run side by side: the
// first is launched plainly, each other one as a programmatic dependent of the
// one before that waits for it only before it ends (kBeside), so that what
// follows the last of them in the stream follows all of them.
enum Follow {
    kPlain = 0,    // after that kernel has ended
    kWait = 1,     // a dependent launch that waits at its start
    kBeside = 2,   // a dependent launch that waits at its end
};
__device__ __forceinline__ void begin_fft(int follow) {
    grid_trigger();
    if (follow == kWait) grid_wait();
}
// (unconditional: it returns at once unless the launch is kBeside, and behind a
// branch the FP64 forward came out 4 to 7 % slower)
__device__ __forceinline__ void end_fft() { grid_wait(); }

template <typename T> inline void set_follow(FwdArgs<T>& a, int f) { a.follow = f; }
template <typename T> inline void set_follow(InvArgs<T>& a, int f) { a.follow = f; }
template <class G> inline void set_follow(G& g, int f) { g.follow = f; }

// One FFT launch; kWait is taken where it pays (short_launch).
template <class... Params, class Args>
cudaError_t fft_launch(void (*kernel)(Params...), const Args& args, dim3 grid, size_t smem,
                       cudaStream_t s, Follow follow) {
    const cudaError_t e = ensure_smem((const void*)kernel, smem);
    if (e) return e;
    if (follow == kWait && !short_launch((long long)grid.x * grid.y)) follow = kPlain;
    Args a = args;
    set_follow(a, follow);
    return launch_kernel(kernel, grid, dim3(kFftThreads), smem, s, follow != kPlain, a);
}

// Iterates idx = tid, tid + kFftThreads, ... as (major, minor) = (idx / d, idx % d)
// without dividing inside the loop.
struct Walk2 {
    int major, minor, step_major, step_minor, d;
    __device__ __forceinline__ Walk2(int start, int d_) : d(d_) {
        major = start / d;
        minor = start - major * d;
        step_major = kFftThreads / d;
        step_minor = kFftThreads - step_major * d;
    }
    __device__ __forceinline__ void next() {
        major += step_major;
        minor += step_minor;
        if (minor >= d) {
            minor -= d;
            ++major;
        }
    }
};

// ---- grouped launches: several plans' rows in one grid ----------------
template <typename T> struct FwdGroup {
    int n, follow;
    int cta_start[kMaxGroup + 1];   // first CTA of each plan
    int nfg[kMaxGroup];             // field groups per latitude of each plan
    FwdArgs<T> a[kMaxGroup];
};

template <typename T> struct InvGroup {
    int n, follow;
    int cta_start[kMaxGroup + 1];
    int nfg[kMaxGroup];
    InvArgs<T> a[kMaxGroup];
};

// ---- reduced grids: a half-length per latitude pair -------------------
// Each CTA takes its latitude pair's FFT shape and the offsets of that
// shape's tables; rows, shared memory and the row pitch are sized for the
// longest row of the grid.
template <typename T> struct RaggedFwd {
    FwdArgs<T> a;
    int follow;
    const RShape* shapes;
    const int* shape_of;
    const int* shift_of;                       // per latitude pair (null: none shifted)
    const typename Vec2<T>::type* shiftbase;   // all shapes' shift phases
    const typename Vec2<T>::type* chirpbase;   // all Bluestein shapes' chirps
    const typename Vec2<T>::type* dftbase;     // all Bluestein shapes' chirp spectra
};

template <typename T> struct RaggedInv {
    InvArgs<T> a;
    int follow;
    const RShape* shapes;
    const int* shape_of;
    const int* shift_of;
    const typename Vec2<T>::type* shiftbase;
    const typename Vec2<T>::type* chirpbase;
    const typename Vec2<T>::type* dftbase;
};

// Per-CTA arguments of a reduced-grid row class: the latitude pair's shape,
// its tables, and its shift.
template <typename Args, typename R>
__device__ __forceinline__ void apply_shape(Args& A, const R& Rg, int jh) {
    const RShape& rs = Rg.shapes[Rg.shape_of[jh]];
    A.shape = rs.sh;
    A.L = rs.L;
    A.twp += rs.tw_off;
    A.twpost += rs.post_off;
    A.rev += rs.rev_off;
    A.shiftph = (Rg.shift_of && Rg.shift_of[jh] && rs.shift_off >= 0)
                    ? Rg.shiftbase + rs.shift_off : nullptr;
    if (rs.bluestein) {
        A.chirp = Rg.chirpbase + rs.chirp_off;
        A.dft = Rg.dftbase + rs.dft_off;
    }
}

// FP32 launches of the kernels in other translation units, and the upload of
// their constant twiddles to the current device.
cudaError_t fft_any_init();
cudaError_t fft_any_forward(const FwdArgs<float>& A, bool strided, dim3 grid, size_t smem,
                            cudaStream_t s,
    Follow follow);
cudaError_t fft_any_inverse(const InvArgs<float>& A, dim3 grid, size_t smem, cudaStream_t s,
    Follow follow);
cudaError_t fft_any_forward_ragged(const RaggedFwd<float>& R, dim3 grid, size_t smem,
                                   cudaStream_t s,
    Follow follow);
cudaError_t fft_any_inverse_ragged(const RaggedInv<float>& R, dim3 grid, size_t smem,
                                   cudaStream_t s,
    Follow follow);
cudaError_t fft_bluestein_init();
cudaError_t fft_bluestein_forward(const RaggedFwd<float>& R, dim3 grid, size_t smem,
                                  cudaStream_t s,
    Follow follow);
cudaError_t fft_bluestein_forward(const RaggedFwd<double>& R, dim3 grid, size_t smem,
                                  cudaStream_t s,
    Follow follow);
cudaError_t fft_bluestein_inverse(const RaggedInv<float>& R, dim3 grid, size_t smem,
                                  cudaStream_t s,
    Follow follow);
cudaError_t fft_bluestein_inverse(const RaggedInv<double>& R, dim3 grid, size_t smem,
                                  cudaStream_t s,
    Follow follow);
cudaError_t fft_group_init();
cudaError_t fft_group_forward(const FwdGroup<float>& G, int ctas, size_t smem, cudaStream_t s,
    Follow follow);
cudaError_t fft_group_inverse(const InvGroup<float>& G, int ctas, size_t smem, cudaStream_t s,
    Follow follow);

// Fixed-point FFT launches of the FP64 path (sht_fft64.cu); the arguments'
// twiddle tables are the fixed-point ones (launch_fixed_twiddles).
cudaError_t fx_forward(const FwdArgs<double>& A, bool strided, dim3 grid, size_t smem,
                       cudaStream_t s,
    Follow follow);
cudaError_t fx_inverse(const InvArgs<double>& A, dim3 grid, size_t smem, cudaStream_t s,
    Follow follow);
cudaError_t fx_forward_ragged(const RaggedFwd<double>& R, dim3 grid, size_t smem, cudaStream_t s,
    Follow follow);
cudaError_t fx_inverse_ragged(const RaggedInv<double>& R, dim3 grid, size_t smem, cudaStream_t s,
    Follow follow);
cudaError_t fx_forward_group(const FwdGroup<double>& G, int ctas, size_t smem, cudaStream_t s,
    Follow follow);
cudaError_t fx_inverse_group(const InvGroup<double>& G, int ctas, size_t smem, cudaStream_t s,
    Follow follow);

}  // namespace sht
