// FFT launches: arguments from the plans, the dispatch on the half-length, and
// the kernels of the compile-time lengths (sht_fft_kernels.h).
#include <limits.h>

#include <algorithm>
#include <mutex>

#include "sht_fft_kernels.h"

namespace sht {
namespace {

template <int LT>
cudaError_t fwd_launch(const FwdArgs<float>& A, bool strided, dim3 grid, size_t smem,
                       cudaStream_t s, Follow follow) {
    if (!strided) return fft_launch(fft_forward_kernel<float, LT, false>, A, grid, smem, s, follow);
    return fft_launch(fft_forward_kernel<float, LT, true>, A, grid, smem, s, follow);
}

template <int LT>
cudaError_t inv_launch(const InvArgs<float>& A, dim3 grid, size_t smem, cudaStream_t s,
                       Follow follow) {
    // Short rows (radices below 16) get a kernel for the plain store alone, its
    // last pass two butterflies at a time: T159 x 256 107.5 -> 104.0 us (6
    // fields per CTA 137 -> 126), T239 x 64 74.7 -> 73.3.  From 512 on it was
    // slower (T639 x 128 777 -> 811, T479 x 64 223 -> 242).
    if constexpr (LT < 512 && inverse_stores_from_last_pass<float, LT>())
        if (A.accumulate == 0)
            return fft_launch(fft_inverse_kernel<float, LT, true>, A, grid, smem, s, follow);
    return fft_launch(fft_inverse_kernel<float, LT>, A, grid, smem, s, follow);
}

// Dispatch on the half-length: the rows of cubic grids (I = 4 (N + 1)) at the
// usual truncations get specialised kernels.  For 64 fields, run-time shape
// -> specialised, forward / inverse us: T479 (L = 960) 280 / 289 -> 205 / 228,
// T383 (768) 188 / 181 -> 140 / 141, T239 (480) 99 / 93 -> 75 / 75, T191 (384)
// 57 / 52 -> 41 / 39.
#define SHT_FFT_DISPATCH(L, CALL, OTHER)   \
    switch (L) {                           \
        case 64: return CALL(64);          \
        case 128: return CALL(128);        \
        case 256: return CALL(256);        \
        case 320: return CALL(320);        \
        case 384: return CALL(384);        \
        case 480: return CALL(480);        \
        case 512: return CALL(512);        \
        case 640: return CALL(640);        \
        case 768: return CALL(768);        \
        case 960: return CALL(960);        \
        case 1024: return CALL(1024);      \
        case 1280: return CALL(1280);      \
        default: return OTHER;             \
    }

cudaError_t fwd_dispatch(const FwdArgs<float>& A, bool strided, dim3 grid, size_t smem,
                         cudaStream_t s, Follow follow) {
#define SHT_FWD(LV) fwd_launch<LV>(A, strided, grid, smem, s, follow)
    SHT_FFT_DISPATCH(A.L, SHT_FWD, fft_any_forward(A, strided, grid, smem, s, follow))
#undef SHT_FWD
}

cudaError_t inv_dispatch(const InvArgs<float>& A, dim3 grid, size_t smem, cudaStream_t s,
                         Follow follow) {
#define SHT_INV(LV) inv_launch<LV>(A, grid, smem, s, follow)
    SHT_FFT_DISPATCH(A.L, SHT_INV, fft_any_inverse(A, grid, smem, s, follow))
#undef SHT_INV
}

template <typename T>
FwdArgs<T> make_fwd_args(const sht_plan_s* p, const void* grid, const RowSource& src,
                         const FwdScale& sc, void* work) {
    using V = typename Vec2<T>::type;
    FwdArgs<T> A;
    A.grid = static_cast<const T*>(grid);
    A.src = src;
    A.work = static_cast<V*>(work);
    A.twp = static_cast<const V*>(p->d_twpass);
    A.twpost = static_cast<const V*>(p->d_twpost);
    A.rev = p->d_rev;
    A.rowscale = sc.rowscale;
    A.mscale0 = sc.mscale0;
    A.mscale1 = sc.mscale1;
    A.colmax = p->d_colmax;
    A.rowoff = nullptr;
    A.jh_list = nullptr;
    A.shiftph = A.chirp = A.dft = nullptr;
    A.F = p->F; A.J = p->J; A.Jh = p->Jh; A.L = p->fft.L; A.N = p->N; A.G = p->G;
    A.LP = fft_row_pitch(p->fft.L, sizeof(T) == 8);
    A.shape = p->fft;
    return A;
}

template <typename T>
cudaError_t fwd_impl(const sht_plan_s* p, const void* grid, const RowSource& src,
                     const FwdScale& sc, void* work, cudaStream_t s) {
    FwdArgs<T> A = make_fwd_args<T>(p, grid, src, sc, work);
    A.src.quads = sizeof(T) == 4 && src.elem_stride == 2 && ((uintptr_t)grid & 15) == 0 &&
                  src.field_stride % 4 == 0 && src.row_stride % 4 == 0 && src.row_offset % 4 == 0;
    if (A.colmax) {
        const cudaError_t e = cudaMemsetAsync(A.colmax, 0, 2 * (size_t)p->F * sizeof(unsigned), s);
        if (e) return e;
    }
    const dim3 g((p->F + p->G - 1) / p->G, p->Jh);
    const bool strided = src.elem_stride != 1;
    if constexpr (sizeof(T) == 8)
        return fx_forward(A, strided, g, p->fft_smem, s, kWait);
    else
        return fwd_dispatch(A, strided, g, p->fft_smem, s, A.colmax ? kPlain : kWait);
}

template <typename T>
InvArgs<T> make_inv_args(const sht_plan_s* p, const void* work, const InvScale& sc,
                         void* grid) {
    using V = typename Vec2<T>::type;
    InvArgs<T> A;
    A.work = static_cast<const V*>(work);
    A.grid = static_cast<T*>(grid);
    A.twp = static_cast<const V*>(p->d_twpass);
    A.twpost = static_cast<const V*>(p->d_twpost);
    A.rev = p->d_rev;
    A.rowscale = sc.rowscale;
    A.mfactor1 = sc.mfactor1;
    A.rowoff = nullptr;
    A.fstride = (long long)p->J * p->I;
    A.jh_list = nullptr;
    A.accumulate = sc.accumulate;
    A.grid2 = static_cast<T*>(sc.grid2);
    A.shiftph = A.chirp = A.dft = nullptr;
    A.F = p->F; A.J = p->J; A.Jh = p->Jh; A.I = p->I; A.L = p->fft.L; A.N = p->N;
    A.G = p->G;
    A.LP = fft_row_pitch(p->fft.L, sizeof(T) == 8);
    A.shape = p->fft;
    return A;
}

template <typename T>
cudaError_t inv_impl(const sht_plan_s* p, const void* work, const InvScale& sc,
                     void* grid, cudaStream_t s) {
    const InvArgs<T> A = make_inv_args<T>(p, work, sc, grid);
    const dim3 g((p->F + p->G - 1) / p->G, p->Jh);
    if constexpr (sizeof(T) == 8)
        return fx_inverse(A, g, p->fft_smem, s, kWait);
    else
        return inv_dispatch(A, g, p->fft_smem, s, kWait);
}

// Arguments of one length class of a reduced grid: that shape's tables and
// row pitch, and the class's latitude-pair list.
template <typename Args>
void set_class(Args& A, const RaggedGrid* rg, const RShape& r, int off, size_t vb) {
    using V = std::remove_cv_t<std::remove_pointer_t<decltype(A.twp)>>;
    A.L = r.sh.L;
    A.shape = r.sh;
    A.LP = fft_row_pitch(r.sh.L, vb == 16);
    A.twp = reinterpret_cast<const V*>(static_cast<const char*>(rg->d_twpass) + r.tw_off * vb);
    A.twpost = reinterpret_cast<const V*>(static_cast<const char*>(rg->d_twpost) + r.post_off * vb);
    A.rev = rg->d_rev + r.rev_off;
    A.jh_list = rg->d_jh + off;
}

template <typename T>
cudaError_t fwd_ragged_class(const FwdArgs<T>& A, dim3 g, size_t smem, cudaStream_t s,
                             Follow follow) {
    if constexpr (sizeof(T) == 8)
        return fx_forward(A, false, g, smem, s, follow);
    else
        return fwd_dispatch(A, false, g, smem, s, follow);
}

template <typename T>
cudaError_t inv_ragged_class(const InvArgs<T>& A, dim3 g, size_t smem, cudaStream_t s,
                             Follow follow) {
    if constexpr (sizeof(T) == 8)
        return fx_inverse(A, g, smem, s, follow);
    else
        return inv_dispatch(A, g, smem, s, follow);
}

// Reduced grid: one launch of the compile-time kernel per length class that
// has one, then one launch of the generic kernel (a shape per CTA) over the
// remaining latitude pairs, then one over the Bluestein rows, side by side
// (a class may be one latitude pair: 8 CTAs of 8 us at octahedral T319 x 64).
template <typename T>
cudaError_t fwd_ragged_impl(const sht_plan_s* p, const void* grid, const FwdScale& sc,
                            void* work, cudaStream_t s) {
    using V = typename Vec2<T>::type;
    const RaggedGrid* rg = p->ragged;
    const size_t vb = sizeof(V);
    RowSource src;
    src.field_stride = rg->npts;
    src.row_stride = 0;
    src.row_offset = 0;
    src.elem_stride = 1;
    FwdArgs<T> base = make_fwd_args<T>(p, grid, src, sc, work);
    base.rowoff = rg->d_rowoff;
    if (base.colmax) {
        const cudaError_t e = cudaMemsetAsync(base.colmax, 0, 2 * (size_t)p->F * sizeof(unsigned), s);
        if (e) return e;
    }
    const unsigned nfg = (p->F + p->G - 1) / p->G;
    Follow follow = kPlain;   // the launches after the first run beside it
    for (const auto& c : rg->classes) {
        FwdArgs<T> A = base;
        set_class(A, rg, rg->h_shapes[c.shape], c.off, vb);
        const cudaError_t e = fwd_ragged_class<T>(A, dim3(nfg, c.count),
                                                  fft_smem_bytes(2 * A.L, p->G, vb == 16), s, follow);
        follow = kBeside;
        if (e) return e;
    }
    RaggedFwd<T> R;
    R.a = base;
    R.a.twp = static_cast<const V*>(rg->d_twpass);
    R.a.twpost = static_cast<const V*>(rg->d_twpost);
    R.a.rev = rg->d_rev;
    R.shapes = rg->d_shapes;
    R.shape_of = rg->d_shape_of;
    R.shift_of = rg->any_shift ? rg->d_shift_of : nullptr;
    R.shiftbase = static_cast<const V*>(rg->d_shiftph);
    R.chirpbase = static_cast<const V*>(rg->d_chirp);
    R.dftbase = static_cast<const V*>(rg->d_dft);
    cudaError_t e;
    if (rg->generic_count > 0) {
        R.a.jh_list = rg->d_jh + rg->generic_off;
        const dim3 g(nfg, rg->generic_count);
        if constexpr (sizeof(T) == 8)
            e = fx_forward_ragged(R, g, p->fft_smem, s, follow);
        else
            e = fft_any_forward_ragged(R, g, p->fft_smem, s, follow);
        if (e) return e;
        follow = kBeside;
    }
    if (rg->blue_count > 0) {
        R.a.jh_list = rg->d_jh + rg->blue_off;
        R.a.G = rg->blue_G;
        const unsigned nfb = (p->F + rg->blue_G - 1) / rg->blue_G;
        e = fft_bluestein_forward(R, dim3(nfb, rg->blue_count), rg->blue_smem, s, follow);
        if (e) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t inv_ragged_impl(const sht_plan_s* p, const void* work, const InvScale& sc,
                            void* grid, cudaStream_t s) {
    using V = typename Vec2<T>::type;
    const RaggedGrid* rg = p->ragged;
    const size_t vb = sizeof(V);
    InvArgs<T> base = make_inv_args<T>(p, work, sc, grid);
    base.rowoff = rg->d_rowoff;
    base.fstride = rg->npts;
    const unsigned nfg = (p->F + p->G - 1) / p->G;
    Follow follow = kPlain;   // the launches after the first run beside it
    for (const auto& c : rg->classes) {
        InvArgs<T> A = base;
        set_class(A, rg, rg->h_shapes[c.shape], c.off, vb);
        const cudaError_t e = inv_ragged_class<T>(A, dim3(nfg, c.count),
                                                  fft_smem_bytes(2 * A.L, p->G, vb == 16), s, follow);
        follow = kBeside;
        if (e) return e;
    }
    RaggedInv<T> R;
    R.a = base;
    R.a.twp = static_cast<const V*>(rg->d_twpass);
    R.a.twpost = static_cast<const V*>(rg->d_twpost);
    R.a.rev = rg->d_rev;
    R.shapes = rg->d_shapes;
    R.shape_of = rg->d_shape_of;
    R.shift_of = rg->any_shift ? rg->d_shift_of : nullptr;
    R.shiftbase = static_cast<const V*>(rg->d_shiftph);
    R.chirpbase = static_cast<const V*>(rg->d_chirp);
    R.dftbase = static_cast<const V*>(rg->d_dft);
    cudaError_t e;
    if (rg->generic_count > 0) {
        R.a.jh_list = rg->d_jh + rg->generic_off;
        const dim3 g(nfg, rg->generic_count);
        if constexpr (sizeof(T) == 8)
            e = fx_inverse_ragged(R, g, p->fft_smem, s, follow);
        else
            e = fft_any_inverse_ragged(R, g, p->fft_smem, s, follow);
        if (e) return e;
        follow = kBeside;
    }
    if (rg->blue_count > 0) {
        R.a.jh_list = rg->d_jh + rg->blue_off;
        R.a.G = rg->blue_G;
        const unsigned nfb = (p->F + rg->blue_G - 1) / rg->blue_G;
        e = fft_bluestein_inverse(R, dim3(nfb, rg->blue_count), rg->blue_smem, s, follow);
        if (e) return e;
    }
    return cudaSuccess;
}

// Fields per CTA of plan q in a grouped launch: its own tuning, else the default
// for the latitudes of all plans together, with half the CTAs (the plans'
// uneven rows fill the gaps: T7 .. T63 x 7 17.2 us with the 124 CTAs of whole
// field groups, 21.0 with 496).
int group_fields(sht_plan_s* const* plans, int n, int q) {
    const sht_plan_s* p = plans[q];
    if (p->tuned) return p->G;
    int pairs = 0;
    for (int i = 0; i < n; ++i) pairs += plans[i]->Jh;
    const bool fp64 = p->prec == SHT_FP64;
    return fft_default_fields(p->I, pairs, p->F, fp64, fft_plan_ctas(fp64) / 2);
}

template <typename T>
cudaError_t fwd_group_impl(sht_plan_s* const* plans, int n, const void* const* grids,
                           cudaStream_t s) {
    FwdGroup<T> G;
    G.n = n;
    G.cta_start[0] = 0;
    size_t smem = 0;
    for (int q = 0; q < n; ++q) {
        const sht_plan_s* p = plans[q];
        RowSource src;
        src.field_stride = (long long)p->J * p->I;
        src.row_stride = p->I;
        src.row_offset = 0;
        src.elem_stride = 1;
        const FwdScale sc{p->d_w_over_I, 1.0, 1.0};
        G.a[q] = make_fwd_args<T>(p, grids[q], src, sc, p->d_work);
        if (p->d_colmax) {
            const cudaError_t e =
                cudaMemsetAsync(p->d_colmax, 0, 2 * (size_t)p->F * sizeof(unsigned), s);
            if (e) return e;
        }
        const int g = G.a[q].G = group_fields(plans, n, q);
        G.nfg[q] = (p->F + g - 1) / g;
        G.cta_start[q + 1] = G.cta_start[q] + G.nfg[q] * p->Jh;
        smem = std::max(smem, fft_smem_bytes(p->I, g, sizeof(T) == 8));
    }
    if constexpr (sizeof(T) == 8)
        return fx_forward_group(G, G.cta_start[n], smem, s, kWait);
    else
        return fft_group_forward(G, G.cta_start[n], smem, s, plans[0]->d_colmax ? kPlain : kWait);
}

template <typename T>
cudaError_t inv_group_impl(sht_plan_s* const* plans, int n, void* const* grids,
                           cudaStream_t s) {
    InvGroup<T> G;
    G.n = n;
    G.cta_start[0] = 0;
    size_t smem = 0;
    for (int q = 0; q < n; ++q) {
        const sht_plan_s* p = plans[q];
        const InvScale sc{nullptr, 1.0};
        G.a[q] = make_inv_args<T>(p, p->d_work, sc, grids[q]);
        const int g = G.a[q].G = group_fields(plans, n, q);
        G.nfg[q] = (p->F + g - 1) / g;
        G.cta_start[q + 1] = G.cta_start[q] + G.nfg[q] * p->Jh;
        smem = std::max(smem, fft_smem_bytes(p->I, g, sizeof(T) == 8));
    }
    if constexpr (sizeof(T) == 8)
        return fx_inverse_group(G, G.cta_start[n], smem, s, kWait);
    else
        return fft_group_inverse(G, G.cta_start[n], smem, s, kWait);
}

}  // namespace

// Write the constant twiddles of the register DFTs to the current device
// (each translation unit with FFT kernels has its own copy).
cudaError_t fft_constants_init() {
    static std::mutex mu;
    static bool done[64] = {false};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
    e = upload_twiddles();
    if (e == cudaSuccess) e = fft_any_init();
    if (e == cudaSuccess) e = fft_bluestein_init();
    if (e == cudaSuccess) e = fft_group_init();
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
    return e;
}

cudaError_t launch_fft_forward_group(sht_plan_s* const* plans, int n,
                                     const void* const* grids, cudaStream_t s) {
    if (plans[0]->prec == SHT_FP64) return fwd_group_impl<double>(plans, n, grids, s);
    return fwd_group_impl<float>(plans, n, grids, s);
}

cudaError_t launch_fft_inverse_group(sht_plan_s* const* plans, int n,
                                     void* const* grids, cudaStream_t s) {
    if (plans[0]->prec == SHT_FP64) return inv_group_impl<double>(plans, n, grids, s);
    return inv_group_impl<float>(plans, n, grids, s);
}

// Factorisation of a half-length for the kernels with run-time shapes.  FP32
// lengths take the passes, out of the register DFT sizes those kernels hold
// (with_radix), with the least estimated time: per pass and value 14
// instructions of shared-memory traffic, twiddles and addresses plus the
// DFT's own, over the share of the CTA's threads that have a butterfly in
// the rounds of its rows.  Two or three passes of large radices then replace
// up to five of 2 .. 8; with few fields (and so rows) in a CTA, small radices
// keep its threads busy (forward / inverse us, L = 288 x 1 field: 12 24
// 18.3 / 16.4, 3 4 4 6 14.7 / 12.3; L = 900 x 1: 30 30 29.9 / 29.1, 9 10 10
// 25.1 / 22.2).
//
// The kernel that holds all those sizes has 128 registers, two CTAs per SM, and
// starts about 1.5 us later than the one of the sizes up to kSmallRadix, which
// has 80 and runs three.  A regular grid of L > 320 takes the latter where the
// instructions that larger radices save, by the estimate, come to less than 20
// million over the grid, or to none.  Sums of the forward and inverse FFT in us,
// all sizes -> up to 10: L = 432 x 4 43.0 -> 28.0, 720 x 1 42.9 -> 27.6, 900 x 2 50.2
// -> 37.0, 360 x 16 53.4 -> 37.1, 1000 x 16 219 -> 202; kept with all sizes: 675 x 8
// 85.9 (109 with up to 10), 1080 x 8 138 (161), 1250 x 8 188 (210).  Shorter rows
// with all sizes take two passes, which is more exact and in grouped launches
// faster (T63 x 67, L = 96: group pair 66.5 us, with three passes 70.3).
FftShape fft_shape(int L, bool fp64, bool compile_time, float* time, int F, int Jh) {
    if (time) *time = 0.f;
    if (fp64 || L == 1 || compile_time) return fft_factor(L, fp64);
    struct Size { int r; float work; };   // instructions of the DFT per value
    static const Size sizes[] = {{2, 1.f}, {3, 3.f}, {4, 2.5f}, {5, 6.f}, {6, 5.3f}, {8, 5.f},
                                 {9, 7.8f}, {10, 8.6f}, {12, 7.5f}, {15, 11.f}, {16, 7.3f},
                                 {20, 10.9f}, {24, 10.3f}, {25, 14.6f}, {30, 14.f}, {32, 10.1f}};
    int g = 16;
    while (g > 1 && (g > F || fft_smem_bytes(2 * L, g, false) > 112 * 1024)) g /= 2;
    auto cost = [&](const Size& z) {
        const int n = 2 * g * (L / z.r), rounds = (n + kFftThreads - 1) / kFftThreads;
        return (14.f + z.work) * (float)(rounds * kFftThreads) / (float)n;
    };
    int best[4], cur[4], nbest = 0;
    float tbest = 0.f;
    auto search = [&](auto&& self, int limit, int rest, int depth, int from, float t) -> void {
        if (rest == 1) {
            if (nbest == 0 || t < tbest) {
                nbest = depth;
                tbest = t;
                for (int i = 0; i < depth; ++i) best[i] = cur[i];
            }
            return;
        }
        if (depth == 4) return;
        for (int i = from; i < (int)(sizeof(sizes) / sizeof(sizes[0])); ++i) {
            if (sizes[i].r > limit || rest % sizes[i].r) continue;
            cur[depth] = sizes[i].r;
            self(self, limit, rest / sizes[i].r, depth + 1, i, t + cost(sizes[i]));
        }
    };
    // instructions per value of the radices found, all threads busy
    auto instructions = [&]() {
        float n = 0.f;
        for (int q = 0; q < nbest; ++q)
            for (const Size& z : sizes) n += best[q] == z.r ? 14.f + z.work : 0.f;
        return n;
    };
    int small[4], nsmall = 0;
    float isaved = 0.f;
    if (Jh > 0 && L > 320) {
        search(search, kSmallRadix, L, 0, 0, 0.f);
        nsmall = nbest;
        for (int q = 0; q < nbest; ++q) small[q] = best[q];
        isaved = instructions();
        nbest = 0;
    }
    search(search, INT_MAX, L, 0, 0, 0.f);
    if (nbest == 0) return fft_factor(L, true);
    if (time) *time = tbest * (float)L;
    isaved -= instructions();
    if (nsmall > 0 && (double)isaved * L * Jh * F < 20e6) {
        nbest = nsmall;
        for (int q = 0; q < nsmall; ++q) best[q] = small[q];
    }
    FftShape sh{};
    sh.L = L;
    sh.npass = nbest;
    // largest first, but 32 (the padding period) last
    std::sort(best, best + nbest, [](int a, int b) {
        return (a == 32 ? 0 : a) > (b == 32 ? 0 : b);
    });
    int span = L, off = 0;
    for (int q = 0; q < nbest; ++q) {
        span /= best[q];
        sh.radix[q] = best[q];
        sh.span[q] = span;
        sh.twoff[q] = off;
        off += (best[q] - 1) * span;
    }
    sh.twtotal = off;
    return sh;
}

size_t bluestein_smem_bytes(int L2, int G, bool fp64) {
    const size_t v = fp64 ? sizeof(double2) : sizeof(float2);
    // rows of length L2 | twiddles of length L2 | column maxima (2 G words)
    return (2 * (size_t)G * fft_row_pitch(L2, fp64) + L2) * v + 8 * (size_t)G;
}

size_t fft_smem_bytes(int I, int G, bool fp64) {
    const size_t L = (size_t)I / 2;
    const size_t rows = 2 * (size_t)G * fft_row_pitch((int)L, fp64);
    // FP64: padded rows + the fields' scales
    if (fp64) return rows * sizeof(double2) + kFxFieldBytes * (size_t)G;
    // FP32: padded rows + per-pass twiddle tables (fewer than L entries) + the
    // column maxima of the forward kernel's output (2 words per field)
    return (rows + L) * sizeof(float2) + 8 * (size_t)G;
}

// The largest power of two that leaves room for the CTAs an SM holds by
// registers (FP32 two, FP64 four) and keeps the grid at 256 (FP64: 512) CTAs
// or more.  A power of two: the threads then divide into whole groups of
// fields and a CTA's workspace pieces into whole sectors (forward / inverse
// us: T319 x 300 bf16x3, 10 fields 443 / 486, 8 fields 370 / 418; T255 x 256,
// 12 fields 229 / 241, 8 fields 206 / 216; Tc479 x 64, 6 fields 402 / 497, 4
// fields 369 / 449).  Small grids (T31 x 32 bf16x3): 16 fields, 66 CTAs
// 10.0 / 11.4, 4 fields, 264 CTAs 8.4 / 8.0; FP64 T63 x 16: 8 fields, 130
// CTAs 18.0 / 22.4, 2 fields, 520 CTAs 15.1 / 14.2.
// A few FP32 fields leave a power of two's last CTA of each latitude with little
// to do.  Up to 5 fields stay together where the latitudes alone fill the grid,
// and up to 12 that make two CTAs are halved (sum of both FFTs, us: T255 x 3, 2
// fields 24.9, 3 20.6; T511 x 3 49.3, 40.4; T255 x 5, 4 fields 27.9, 5 22.9; T199 x
// 9, 8 fields 49.7, 5 37.2; T255 x 12, 8 fields 36.7, 6 35.6; T319 x 12 the other
// way, 52.0 and 54.6).
int fft_default_fields(int I, int Jh, int F, bool fp64, int ctas) {
    const size_t budget = (fp64 ? 55 : 112) * 1024;
    int g = 16;
    while (g > 1 && (g > F || fft_smem_bytes(I, g, fp64) > budget ||
                     (long)Jh * ((F + g - 1) / g) < ctas))
        g /= 2;
    if (!fp64) {
        if (F <= 5 && Jh >= ctas && fft_smem_bytes(I, F, false) <= budget)
            g = F;
        else if (F <= 12 && (F + g - 1) / g == 2)
            g = (F + 1) / 2;
    }
    return fft_smem_bytes(I, g, fp64) <= 227 * 1024 ? g : 0;
}

cudaError_t launch_fft_forward(const sht_plan_s* p, const void* grid,
                               const RowSource& src, const FwdScale& sc,
                               void* work, cudaStream_t s) {
    if (p->ragged) {
        if (p->prec == SHT_FP64) return fwd_ragged_impl<double>(p, grid, sc, work, s);
        return fwd_ragged_impl<float>(p, grid, sc, work, s);
    }
    if (p->prec == SHT_FP64) return fwd_impl<double>(p, grid, src, sc, work, s);
    return fwd_impl<float>(p, grid, src, sc, work, s);
}

cudaError_t launch_fft_inverse(const sht_plan_s* p, const void* work,
                               const InvScale& sc, void* grid, cudaStream_t s) {
    if (p->ragged) {
        if (p->prec == SHT_FP64) return inv_ragged_impl<double>(p, work, sc, grid, s);
        return inv_ragged_impl<float>(p, work, sc, grid, s);
    }
    if (p->prec == SHT_FP64) return inv_impl<double>(p, work, sc, grid, s);
    return inv_impl<float>(p, work, sc, grid, s);
}

}  // namespace sht
