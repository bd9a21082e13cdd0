// FFT kernel templates, included by the translation units that instantiate
// them: sht_fft.cu (compile-time lengths), sht_fft_any.cu (shapes known at
// run time), sht_fft_bluestein.cu and sht_fft_group.cu.
// Batched real FFT along latitude circles, fused with the equatorial
// parity fold (Appendix B) and the [m][parity][j][field] layout change that
// the per-m Legendre contraction wants.
//
// A row of I real samples x_i is read as L = I/2 complex values
// z_k = x_{2k} + i x_{2k+1}; an in-place mixed-radix decimation-in-
// frequency FFT of length L runs in shared memory and leaves Z in
// digit-reversed order (rev(k) = position of frequency k).  The real
// spectrum follows from
//   X_m = (Z_m + conj Z_{L-m})/2 + e^{-2 pi i m/I} (Z_m - conj Z_{L-m})/(2i).
// The inverse builds Z_q = (Y_q + conj Y_{L-q}) + i e^{+2 pi i q/I} (Y_q - conj Y_{L-q})
// from the Hermitian spectrum Y (Y_0 real, Y_m = 0 for m > N) and runs the
// same forward FFT on conj(Z): z = conj(FFT(conj Z)), x_{2k} = Re z_k,
// x_{2k+1} = Im z_k.
//
// One CTA owns latitude pair (j, J-1-j) (0-based; the Equator row alone)
// for G consecutive fields: 2G rows of L complex values plus the per-pass
// twiddle tables in shared memory.  Rows use the padded layout of
// PadShift (element pos at pos + (pos >> s), odd row pitch), which keeps the
// passes' power-of-two strides, the digit-reversed accesses and the
// row-to-row distance off a single bank; each pass reads its twiddles from
// a table contiguous in the butterfly index.  Global loads are
// asynchronous element copies (cp.async) straight into the padded layout,
// all in flight before the CTA waits once, except where the FP32 two-pass
// lengths (L = Q x 32, Q >= 8) let the forward's first pass read the grid
// rows into registers and the inverse's last pass write them from
// registers.  The CTAs of all field groups of one latitude are adjacent in
// the launch order, so their partial-sector writes of the same workspace
// rows meet in L2.
//
// The half-lengths of the standard grids (fft_has_fixed_kernel) have kernels
// specialised at compile time: radices, spans, twiddle offsets and the
// digit reversal are constants, so the index arithmetic needs no integer
// division by a runtime value.  Other lengths use the same code with the
// shape read at run time: two to four passes of register DFT sizes up to 32,
// chosen at plan creation (fft_shape), the forward's first pass reading the
// grid rows and the inverse's last pass writing them.  Passes of radices 8,
// 4, 2, 3, 5 through shared memory took 1.2 to 1.8 times as long (forward /
// inverse us for 64 fields: T399, L = 800, 281 / 329 -> 207 / 207; T179, L = 360,
// 81 / 82 -> 53 / 50; T119, L = 240, 51 / 46 -> 30 / 29).
// Grouped launches branch per CTA to the body of their plan's length (64, 128,
// 256, 320, 512, 640, 1024, 1280; the run-time body for the others), and a
// reduced grid launches the compile-time kernel once per row length it
// contains, over a list of latitude pairs.
#pragma once

#include <math.h>

#include <type_traits>

#include "sht_fft_common.h"
#include "sht_internal.h"

namespace sht {
namespace {

constexpr int NT = kFftThreads;

// Paired FP32 arithmetic (add/sub/mul.f32x2): one instruction on both
// components of a complex value.
__device__ __forceinline__ float2 add_f32x2(float2 a, float2 b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(*reinterpret_cast<const uint64_t*>(&a)), "l"(*reinterpret_cast<const uint64_t*>(&b)));
    return *reinterpret_cast<const float2*>(&d);
}
__device__ __forceinline__ float2 sub_f32x2(float2 a, float2 b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(*reinterpret_cast<const uint64_t*>(&a)), "l"(*reinterpret_cast<const uint64_t*>(&b)));
    return *reinterpret_cast<const float2*>(&d);
}
__device__ __forceinline__ float2 mul_f32x2(float2 a, float2 b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(d)
        : "l"(*reinterpret_cast<const uint64_t*>(&a)), "l"(*reinterpret_cast<const uint64_t*>(&b)));
    return *reinterpret_cast<const float2*>(&d);
}

template <typename T> struct C2 {
    using V = typename Vec2<T>::type;
    static __device__ __forceinline__ V make(T x, T y) { V v; v.x = x; v.y = y; return v; }
    static __device__ __forceinline__ V add(V a, V b) {
        if constexpr (sizeof(T) == 4)
            return add_f32x2(a, b);
        else
            return make(a.x + b.x, a.y + b.y);
    }
    static __device__ __forceinline__ V sub(V a, V b) {
        if constexpr (sizeof(T) == 4)
            return sub_f32x2(a, b);
        else
            return make(a.x - b.x, a.y - b.y);
    }
    static __device__ __forceinline__ V mul(V a, V b) {
        return make(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
    }
    static __device__ __forceinline__ V conj(V a) { return make(a.x, -a.y); }
    static __device__ __forceinline__ V scale(V a, T s) {
        if constexpr (sizeof(T) == 4)
            return mul_f32x2(a, make(s, s));
        else
            return make(a.x * s, a.y * s);
    }
    // multiply by -i
    static __device__ __forceinline__ V mul_mi(V a) { return make(a.y, -a.x); }
    // multiply by +i
    static __device__ __forceinline__ V mul_pi(V a) { return make(-a.y, a.x); }
};

// W_N^e = exp(-2 pi i e/N) for the composite register DFT sizes whose factors
// are not coprime, written once per device by fft_constants_init.
constexpr int kComposite[] = {9, 16, 25, 32};
constexpr int tw_offset(int n) {
    int off = 0;
    for (int c : kComposite) {
        if (c == n) return off;
        off += c;
    }
    return off;
}
constexpr int kTwTotal = tw_offset(0);
__constant__ float2 c_twf[kTwTotal];

// ---- radix-R DFTs (forward sign) ---------------------------------------
template <typename T, int R> struct Dft;

template <typename T> struct Dft<T, 2> {
    using V = typename Vec2<T>::type;
    static __device__ __forceinline__ constexpr int pos(int k) { return k; }
    static __device__ __forceinline__ void run(V* a) {
        using K = C2<T>;
        const V y0 = K::add(a[0], a[1]);
        a[1] = K::sub(a[0], a[1]);
        a[0] = y0;
    }
};

template <typename T> struct Dft<T, 3> {
    using V = typename Vec2<T>::type;
    static __device__ __forceinline__ constexpr int pos(int k) { return k; }
    static __device__ __forceinline__ void run(V* a) {
        using K = C2<T>;
        const T h = (T)0.86602540378443864676;   // sin(2 pi/3)
        const V t1 = K::add(a[1], a[2]), t2 = K::sub(a[1], a[2]);
        const V y0 = K::add(a[0], t1);
        const V m0 = K::make(a[0].x - (T)0.5 * t1.x, a[0].y - (T)0.5 * t1.y);
        // m0 -+ i h t2, component by component
        a[0] = y0;
        a[1] = K::make(m0.x + h * t2.y, m0.y - h * t2.x);
        a[2] = K::make(m0.x - h * t2.y, m0.y + h * t2.x);
    }
};

template <typename T> struct Dft<T, 4> {
    using V = typename Vec2<T>::type;
    static __device__ __forceinline__ constexpr int pos(int k) { return k; }
    static __device__ __forceinline__ void run(V* a) {
        using K = C2<T>;
        const V s02 = K::add(a[0], a[2]), d02 = K::sub(a[0], a[2]);
        const V s13 = K::add(a[1], a[3]), t = K::sub(a[1], a[3]);
        a[0] = K::add(s02, s13);
        a[2] = K::sub(s02, s13);
        // d02 -+ i t, component by component (no swapped pair)
        a[1] = K::make(d02.x + t.y, d02.y - t.x);
        a[3] = K::make(d02.x - t.y, d02.y + t.x);
    }
};

template <typename T> struct Dft<T, 8> {
    using V = typename Vec2<T>::type;
    static __device__ __forceinline__ constexpr int pos(int k) { return k; }
    static __device__ __forceinline__ void run(V* a) {
        using K = C2<T>;
        const T r = (T)0.70710678118654752440;   // 1/sqrt(2)
        // even and odd halves by radix 4, then y_k = E_k + W8^k O_k,
        // y_{k+4} = E_k - W8^k O_k with W8 = e^{-2 pi i/8}
        V e[4] = {a[0], a[2], a[4], a[6]};
        V o[4] = {a[1], a[3], a[5], a[7]};
        Dft<T, 4>::run(e);
        Dft<T, 4>::run(o);
        const V o1 = K::make(r * (o[1].x + o[1].y), r * (o[1].y - o[1].x));   // W8^1 o1
        const V o3 = K::make(r * (o[3].y - o[3].x), -r * (o[3].x + o[3].y));   // W8^3 o3
        a[0] = K::add(e[0], o[0]);
        a[4] = K::sub(e[0], o[0]);
        a[1] = K::add(e[1], o1);
        a[5] = K::sub(e[1], o1);
        // W8^2 o2 = -i o2, component by component
        a[2] = K::make(e[2].x + o[2].y, e[2].y - o[2].x);
        a[6] = K::make(e[2].x - o[2].y, e[2].y + o[2].x);
        a[3] = K::add(e[3], o3);
        a[7] = K::sub(e[3], o3);
    }
};

template <typename T> struct Dft<T, 5> {
    using V = typename Vec2<T>::type;
    static __device__ __forceinline__ constexpr int pos(int k) { return k; }
    static __device__ __forceinline__ void run(V* a) {
        using K = C2<T>;
        // cos/sin of 2 pi/5 and 4 pi/5
        const T c1 = (T)0.30901699437494742410, c2 = (T)-0.80901699437494742410;
        const T s1 = (T)0.95105651629515357212, s2 = (T)0.58778525229247312917;
        const V b1 = K::add(a[1], a[4]), d1 = K::sub(a[1], a[4]);
        const V b2 = K::add(a[2], a[3]), d2 = K::sub(a[2], a[3]);
        const V y0 = K::add(a[0], K::add(b1, b2));
        const V p1 = K::make(a[0].x + c1 * b1.x + c2 * b2.x, a[0].y + c1 * b1.y + c2 * b2.y);
        const V p2 = K::make(a[0].x + c2 * b1.x + c1 * b2.x, a[0].y + c2 * b1.y + c1 * b2.y);
        // q1 = s1 d1 + s2 d2, q2 = s2 d1 - s1 d2; y1 = p1 - i q1, y4 = p1 + i q1,
        // y2 = p2 - i q2, y3 = p2 + i q2
        const V q1 = K::make(s1 * d1.x + s2 * d2.x, s1 * d1.y + s2 * d2.y);
        const V q2 = K::make(s2 * d1.x - s1 * d2.x, s2 * d1.y - s1 * d2.y);
        a[0] = y0;
        a[1] = K::make(p1.x + q1.y, p1.y - q1.x);
        a[4] = K::make(p1.x - q1.y, p1.y + q1.x);
        a[2] = K::make(p2.x + q2.y, p2.y - q2.x);
        a[3] = K::make(p2.x - q2.y, p2.y + q2.x);
    }
};

// Composite DFT of size N = A B in registers, in place:
//   X[k1 + A k2] = sum_b W_B^{b k2} W_N^{b k1} sum_a x[b + B a] W_A^{a k1},
// i.e. B DFTs of size A over stride-B subsequences (results written back to
// the same registers), the twiddles W_N^{b k1} (constant memory), then A
// DFTs of size B over each contiguous block of B.  X[k] is left in
// register pos(k) = k1 B + k2 (k = k1 + A k2); the butterfly stores with
// this map, so no register array beyond the input is live.  A is a basic
// size (results in order); B may be composite itself.
template <typename T, int A, int B>
struct DftComposite {
    using V = typename Vec2<T>::type;
    static constexpr int TWOFF = tw_offset(A * B);
    static __device__ __forceinline__ constexpr int pos(int k) {
        return (k % A) * B + Dft<T, B>::pos(k / A);
    }
    static __device__ __forceinline__ void run(V* x) {
        using K = C2<T>;
        constexpr int N = A * B;
#pragma unroll
        for (int b = 0; b < B; ++b) {
            V t[A];
#pragma unroll
            for (int a = 0; a < A; ++a) t[a] = x[b + B * a];
            Dft<T, A>::run(t);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1)
                x[b + B * k1] =
                    (b * k1 == 0) ? t[k1] : K::mul(t[k1], c_twf[TWOFF + (b * k1) % N]);
        }
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            V t[B];
#pragma unroll
            for (int b = 0; b < B; ++b) t[b] = x[k1 * B + b];
            Dft<T, B>::run(t);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) x[k1 * B + k2] = t[k2];
        }
    }
};

// The same for coprime A and B by the Good-Thomas index maps: with
// n = B n1 + A n2 (mod N), W_N^{n k} = W_A^{n1 k} W_B^{n2 k}, so
//   X[k] = sum_n2 W_B^{n2 (k mod B)} sum_n1 W_A^{n1 (k mod A)} x[n]
// needs no twiddles (a size 40 saves 28 complex products of 4 instructions
// and their rounding); the maps only name registers.
template <typename T, int A, int B>
struct DftCoprime {
    using V = typename Vec2<T>::type;
    static constexpr int N = A * B;
    static __device__ __forceinline__ constexpr int pos(int k) {
        return (B * (k % A) + A * Dft<T, B>::pos(k % B)) % N;
    }
    static __device__ __forceinline__ void run(V* x) {
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) {
            V t[A];
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) t[n1] = x[(B * n1 + A * n2) % N];
            Dft<T, A>::run(t);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) x[(B * k1 + A * n2) % N] = t[k1];
        }
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            V t[B];
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) t[n2] = x[(B * k1 + A * n2) % N];
            Dft<T, B>::run(t);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) x[(B * k1 + A * k2) % N] = t[k2];
        }
    }
};

template <typename T> struct Dft<T, 6> : DftCoprime<T, 2, 3> {};
template <typename T> struct Dft<T, 9> : DftComposite<T, 3, 3> {};
template <typename T> struct Dft<T, 10> : DftCoprime<T, 2, 5> {};
template <typename T> struct Dft<T, 12> : DftCoprime<T, 4, 3> {};
template <typename T> struct Dft<T, 15> : DftCoprime<T, 3, 5> {};
template <typename T> struct Dft<T, 16> : DftComposite<T, 4, 4> {};
template <typename T> struct Dft<T, 20> : DftCoprime<T, 4, 5> {};
template <typename T> struct Dft<T, 24> : DftCoprime<T, 8, 3> {};
template <typename T> struct Dft<T, 25> : DftComposite<T, 5, 5> {};
template <typename T> struct Dft<T, 30> : DftCoprime<T, 5, 6> {};
template <typename T> struct Dft<T, 32> : DftComposite<T, 8, 4> {};
template <typename T> struct Dft<T, 40> : DftCoprime<T, 8, 5> {};

// f(integral_constant<int, r>) for a radix known at run time: FP64 (Bluestein
// rows) 2, 3, 4, 5 and 8, FP32 the register DFT sizes up to kSmallRadix, with
// ALL every one.
template <typename T, bool ALL, class F>
__device__ __forceinline__ void with_radix(int r, F f) {
#define SHT_RADIX(R) \
    case R: f(std::integral_constant<int, R>{}); return;
    if constexpr (sizeof(T) == 4 && ALL) {
        switch (r) {
            SHT_RADIX(2) SHT_RADIX(3) SHT_RADIX(4) SHT_RADIX(5) SHT_RADIX(6)
            SHT_RADIX(9) SHT_RADIX(10) SHT_RADIX(12) SHT_RADIX(15) SHT_RADIX(16)
            SHT_RADIX(20) SHT_RADIX(24) SHT_RADIX(25) SHT_RADIX(30) SHT_RADIX(32)
            default: break;
        }
    } else if constexpr (sizeof(T) == 4) {
        switch (r) {
            SHT_RADIX(2) SHT_RADIX(3) SHT_RADIX(4) SHT_RADIX(5) SHT_RADIX(6)
            SHT_RADIX(9) SHT_RADIX(10)
            default: break;
        }
    } else {
        switch (r) {
            SHT_RADIX(2) SHT_RADIX(3) SHT_RADIX(4) SHT_RADIX(5)
            default: break;
        }
    }
    f(std::integral_constant<int, 8>{});
#undef SHT_RADIX
}

// One DIF butterfly of radix R: reads z[base + t M], t < R, applies the
// radix-R DFT, multiplies output k1 by W_S^{n1 k1} (per-pass table entry
// (k1 - 1) M + n1) and writes it back to z[base + k1 M].
template <typename T, int R>
__device__ __forceinline__ void bfly(typename Vec2<T>::type* z, int base, int M,
                                     const typename Vec2<T>::type* tw, int n1) {
    using V = typename Vec2<T>::type;
    using K = C2<T>;
    V a[R];
#pragma unroll
    for (int t = 0; t < R; ++t) a[t] = z[ph<T>(base + t * M)];
    Dft<T, R>::run(a);
    // output k1 sits in register pos(k1)
    if (n1 != 0) {
#pragma unroll
        for (int k1 = 1; k1 < R; ++k1) {
            a[Dft<T, R>::pos(k1)] = K::mul(a[Dft<T, R>::pos(k1)], tw[(k1 - 1) * M + n1]);
        }
    }
#pragma unroll
    for (int k1 = 0; k1 < R; ++k1) z[ph<T>(base + k1 * M)] = a[Dft<T, R>::pos(k1)];
}

// The same with the span M a compile-time constant.  When M is a multiple
// of the padding period P (pad one element per P), or R M divides P, the
// padded positions of the R elements are ph(base) + t STEP with a constant
// STEP, so one padded index serves the whole butterfly.
template <typename T, int R, int M>
__device__ __forceinline__ void bfly_fixed(typename Vec2<T>::type* z, int base,
                                           const typename Vec2<T>::type* tw, int n1) {
    using V = typename Vec2<T>::type;
    using K = C2<T>;
    constexpr int P = 1 << PadShift<T>::value;
    if constexpr (M % P == 0 || P % (R * M) == 0) {
        constexpr int STEP = (M % P == 0) ? M + M / P : M;
        V* zb = z + ph<T>(base);
        V a[R];
#pragma unroll
        for (int t = 0; t < R; ++t) a[t] = zb[t * STEP];
        Dft<T, R>::run(a);
        if (M > 1 && n1 != 0) {
#pragma unroll
            for (int k1 = 1; k1 < R; ++k1)
                a[Dft<T, R>::pos(k1)] = K::mul(a[Dft<T, R>::pos(k1)], tw[(k1 - 1) * M + n1]);
        }
#pragma unroll
        for (int k1 = 0; k1 < R; ++k1) zb[k1 * STEP] = a[Dft<T, R>::pos(k1)];
    } else {
        bfly<T, R>(z, base, M, tw, n1);
    }
}

// In-place mixed-radix DIF FFT over `nrows` padded rows (pitch LP), passes
// p0 .. p1 - 1 of a shape known at run time.
template <typename T, bool ALL>
__device__ __forceinline__ void passes_runtime(typename Vec2<T>::type* rows, int nrows, int LP,
                                               const FftShape& sh, int p0, int p1,
                                               const typename Vec2<T>::type* twp) {
    for (int p = p0; p < p1; ++p) {
        const int M = sh.span[p];
        const typename Vec2<T>::type* tw = twp + sh.twoff[p];
        with_radix<T, ALL>(sh.radix[p], [&](auto rc) {
            constexpr int R = decltype(rc)::value;
            const int nb = sh.L / R, S = R * M;
            for (int idx = threadIdx.x; idx < nrows * nb; idx += NT) {
                const int row = idx / nb, b = idx - row * nb;
                const int blk = b / M, n1 = b - blk * M;
                bfly<T, R>(rows + (size_t)row * LP, blk * S + n1, M, tw, n1);
            }
        });
        __syncthreads();
    }
}

// The same with the shape a compile-time constant (passes P .. END-1).
template <typename T, int L, int P, int END = FacOf<L, sizeof(T) == 8>::v.npass>
__device__ __forceinline__ void passes_fixed(typename Vec2<T>::type* rows, int nrows, int LP,
                                             const typename Vec2<T>::type* twp) {
    constexpr FftShape F = FacOf<L, sizeof(T) == 8>::v;
    if constexpr (P < END) {
        constexpr int R = F.radix[P];
        constexpr int M = F.span[P];
        constexpr int S = R * M;
        constexpr int NB = L / R;
        constexpr int OFF = F.twoff[P];
        const int total = nrows * NB;
        for (int idx = threadIdx.x; idx < total; idx += NT) {
            const int row = idx / NB;
            const int b = idx - row * NB;
            const int blk = b / M;
            const int n1 = b - blk * M;
            bfly_fixed<T, R, M>(rows + (size_t)row * LP, blk * S + n1, twp + OFF, n1);
        }
        __syncthreads();
        passes_fixed<T, L, P + 1, END>(rows, nrows, LP, twp);
    }
}

// FP32 two-pass shapes L = Q x 32 with Q >= 8: the forward runs its first
// pass from the grid rows (below), the inverse its last pass into them.
template <typename T, int L>
__host__ __device__ constexpr bool first_pass_from_global() {
    if constexpr (sizeof(T) != 4 || L <= 0) {
        return false;
    } else {
        constexpr FftShape F = FacOf<L, false>::v;
        return F.npass == 2 && F.radix[1] == 32 && F.span[0] == 32 && F.radix[0] >= 8;
    }
}

// FP32 two-pass shapes L = Q x 32 with Q >= 8: the inverse runs its last
// pass (radix 32, span 1) straight into the grid rows.  Butterfly b of a
// row holds frequencies b + Q k1 (k1 < 32) of the digit-reversed output,
// so for each k1 the lanes of a warp store consecutive complex values
// (at least 64 contiguous bytes), and the result needs no shared-memory
// round trip before the store.
template <typename T, int L>
__host__ __device__ constexpr bool inverse_stores_from_last_pass() {
    if constexpr (sizeof(T) != 4 || L <= 0) {
        return false;
    } else {
        constexpr FftShape F = FacOf<L, false>::v;
        return F.npass == 2 && F.radix[1] == 32 && F.radix[0] >= 8;
    }
}

// LT > 0: the compile-time shape of that half-length; LT = -1: any shape at
// run time; LT = -3: any shape of radices up to kSmallRadix.
template <typename T, int LT>
__device__ __forceinline__ void run_passes(typename Vec2<T>::type* rows, int nrows, int LP,
                                           const FftShape& sh,
                                           const typename Vec2<T>::type* twp) {
    if constexpr (LT > 0)
        passes_fixed<T, LT, 0>(rows, nrows, LP, twp);
    else
        passes_runtime<T, LT == -1>(rows, nrows, LP, sh, 0, sh.npass, twp);
}

// Bluestein's chirp-z DFT of rows of half-length L (any L), for the rows of
// reduced grids whose L has a prime factor above 5.  With
// c_n = e^{-i pi n^2 / L},
//   Z_k = sum_n z_n e^{-2 pi i n k / L} = c_k sum_n (z_n c_n) conj(c_{k-n}),
// a circular convolution of length L2 >= 2L - 1 (sh.L, 2-3-5-smooth) of
// a_n = z_n c_n (zero-padded) with the conjugate chirp wrapped around L2,
// whose DFT D (divided by L2) is a table:
//   Z_k = c_k conj(r_k),  r = DFT(conj(DFT(a) D)).
// In place on nrows padded rows at once: on entry a, on return r, both in
// natural order.  The first DFT runs its passes forwards (decimation in
// frequency) and leaves the digit-reversed order; the second runs the
// transposed passes backwards (decimation in time), which takes that order
// back to the natural one, so nothing is permuted.  The last pass of the
// first and the first of the second work on the same R contiguous values
// (span 1): one butterfly in registers does both, with the product by D
// between (D in the order in which the threads read it, see
// bluestein_dft_kernel).
template <typename T>
__device__ __noinline__ void bluestein_rows(typename Vec2<T>::type* rows, int nrows, int LP,
                                            const FftShape& sh,
                                            const typename Vec2<T>::type* tws,
                                            const typename Vec2<T>::type* dft) {
    using V = typename Vec2<T>::type;
    using K = C2<T>;
    const int np = sh.npass;
    passes_runtime<T, true>(rows, nrows, LP, sh, 0, np - 1, tws);
    with_radix<T, true>(sh.radix[np - 1], [&](auto rc) {
        constexpr int R = decltype(rc)::value;
        const int nb = sh.L / R;
        for (int idx = threadIdx.x; idx < nrows * nb; idx += NT) {
            const int row = idx / nb, b = idx - row * nb;
            V* z = rows + (size_t)row * LP;
            V a[R], y[R];
#pragma unroll
            for (int t = 0; t < R; ++t) a[t] = z[ph<T>(b * R + t)];
            Dft<T, R>::run(a);
#pragma unroll
            for (int t = 0; t < R; ++t)
                y[t] = K::conj(K::mul(a[Dft<T, R>::pos(t)], dft[t * nb + b]));
            Dft<T, R>::run(y);
#pragma unroll
            for (int t = 0; t < R; ++t) z[ph<T>(b * R + t)] = y[Dft<T, R>::pos(t)];
        }
    });
    __syncthreads();
    for (int p = np - 2; p >= 0; --p) {
        const int M = sh.span[p];
        const V* tw = tws + sh.twoff[p];
        with_radix<T, true>(sh.radix[p], [&](auto rc) {
            constexpr int R = decltype(rc)::value;
            const int nb = sh.L / R, S = R * M;
            for (int idx = threadIdx.x; idx < nrows * nb; idx += NT) {
                const int row = idx / nb, b = idx - row * nb;
                const int blk = b / M, n1 = b - blk * M, at = blk * S + n1;
                V* z = rows + (size_t)row * LP;
                V a[R];
#pragma unroll
                for (int t = 0; t < R; ++t) a[t] = z[ph<T>(at + t * M)];
                if (n1 != 0) {
#pragma unroll
                    for (int t = 1; t < R; ++t) a[t] = K::mul(a[t], tw[(t - 1) * M + n1]);
                }
                Dft<T, R>::run(a);
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) z[ph<T>(at + k1 * M)] = a[Dft<T, R>::pos(k1)];
            }
        });
        __syncthreads();
    }
}

extern __shared__ __align__(16) unsigned char fft_smem_raw[];

template <typename T, int LT, bool STRIDED>
__device__ __forceinline__ void fwd_body(const FwdArgs<T>& A, int fg, int jh) {
    using V = typename Vec2<T>::type;
    using K = C2<T>;
    const int L = LT > 0 ? LT : A.L;
    const int LP = LT == -2 ? row_pitch<T>(A.shape.L) : A.LP;
    V* rows = reinterpret_cast<V*>(fft_smem_raw);
    V* tws = rows + (size_t)2 * A.G * LP;
    const int f0 = fg * A.G;
    const int nf = min(A.G, A.F - f0);
    const bool equator = (jh == A.Jh - 1);
    const int nrows = equator ? nf : 2 * nf;
    const int tid = threadIdx.x;
    auto row_ptr = [&](int r) -> const T* {
        const int f = f0 + (r < nf ? r : r - nf);
        const int j = (r < nf) ? jh : (A.J - 1 - jh);
        if (A.rowoff) return A.grid + (long long)f * A.src.field_stride + A.rowoff[j];
        return A.grid + (long long)f * A.src.field_stride + A.src.row_offset +
               (long long)j * A.src.row_stride;
    };

    // Complex element k of a row straight from the grid.  In a nested fine grid
    // of twice the longitudes one 16-byte load holds the two samples wanted and
    // the two between (T511 -> T255 x 64: 88 -> 76 us); larger strides are copied
    // to shared memory first (as two loads into registers T1279 -> T319 x 64 took
    // 199 us against 185).
    auto load_z = [&](const V* x, int k) -> V {
        if constexpr (!STRIDED) {
            return x[k];
        } else {
            const float4 v = reinterpret_cast<const float4*>(x)[k];
            return K::make((T)v.x, (T)v.z);
        }
    };
    const bool direct = !STRIDED || A.src.quads;
    if (first_pass_from_global<T, LT>() && direct) {
        if constexpr (first_pass_from_global<T, LT>()) {
            // The first pass (radix Q, span 32) reads its inputs straight from
            // the grid rows into registers: butterfly n1 of a row takes
            // z[n1 + 32 t], t < Q, so for each t the lanes of a warp load 256
            // contiguous bytes.  Only the twiddle table is copied
            // asynchronously; the first butterfly's loads are in flight while
            // the CTA waits for it.
            constexpr FftShape FS = FacOf<LT, false>::v;
            constexpr int Q = FS.radix[0];
            constexpr int M = FS.span[0];                                  // 32
            constexpr int STEP = M + (M >> PadShift<T>::value);            // padded
            load_twiddles_async(tws, A.twp, FS.twtotal);
            const int total = nrows * M;
            V a[Q];
            auto load = [&](int idx) {
                const int r = idx / M, n1 = idx - r * M;
                const V* x = reinterpret_cast<const V*>(row_ptr(r));
#pragma unroll
                for (int t = 0; t < Q; ++t) a[t] = load_z(x, n1 + t * M);
            };
            auto finish = [&](int idx) {
                const int r = idx / M, n1 = idx - r * M;
                Dft<T, Q>::run(a);
                if (n1 != 0) {
#pragma unroll
                    for (int k1 = 1; k1 < Q; ++k1)
                        a[Dft<T, Q>::pos(k1)] =
                            K::mul(a[Dft<T, Q>::pos(k1)], tws[(k1 - 1) * M + n1]);
                }
                V* zb = rows + (size_t)r * LP + n1;
#pragma unroll
                for (int k1 = 0; k1 < Q; ++k1) zb[k1 * STEP] = a[Dft<T, Q>::pos(k1)];
            };
            if (tid < total) load(tid);
            cp_async_wait_all();
            __syncthreads();
            if (tid < total) finish(tid);
            for (int idx = tid + NT; idx < total; idx += NT) {
                load(idx);
                finish(idx);
            }
            __syncthreads();
            passes_fixed<T, LT, 1>(rows, nrows, LP, tws);
        }
    } else if ((LT == -1 || LT == -3) && sizeof(T) == 4 && A.shape.npass > 0 && direct) {
        // the same with the shape known at run time
        const int M = A.shape.span[0];
        load_twiddles_async(tws, A.twp, A.shape.twtotal);
        with_radix<T, LT == -1>(A.shape.radix[0], [&](auto rc) {
            constexpr int R = decltype(rc)::value;
            const int total = nrows * M;
            bool waited = false;
            for (int idx = tid; idx < total || !waited; idx += NT) {
                const bool work = idx < total;
                const int r = work ? idx / M : 0, n1 = idx - r * M;
                V a[R];
                if (work) {
                    const V* x = reinterpret_cast<const V*>(row_ptr(r));
#pragma unroll
                    for (int t = 0; t < R; ++t) a[t] = load_z(x, n1 + t * M);
                }
                if (!waited) {
                    cp_async_wait_all();
                    __syncthreads();
                    waited = true;
                }
                if (!work) break;
                Dft<T, R>::run(a);
                if (n1 != 0) {
#pragma unroll
                    for (int k1 = 1; k1 < R; ++k1)
                        a[Dft<T, R>::pos(k1)] =
                            K::mul(a[Dft<T, R>::pos(k1)], tws[(k1 - 1) * M + n1]);
                }
                V* zb = rows + (size_t)r * LP;
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) zb[ph<T>(n1 + k1 * M)] = a[Dft<T, R>::pos(k1)];
            }
        });
        __syncthreads();
        passes_runtime<T, LT == -1>(rows, nrows, LP, A.shape, 1, A.shape.npass, tws);
    } else if constexpr (LT == -2) {
        load_twiddles_async(tws, A.twp, A.shape.twtotal);
        for (int r = 0; r < nrows; ++r) {
            const V* x = reinterpret_cast<const V*>(row_ptr(r));
            V* d = rows + (size_t)r * LP;
            for (int n = tid; n < A.shape.L; n += NT)
                d[ph<T>(n)] = n < L ? K::mul(x[n], A.chirp[n]) : K::make((T)0, (T)0);
        }
        cp_async_wait_all();
        __syncthreads();
        bluestein_rows<T>(rows, nrows, LP, A.shape, tws, A.dft);
    } else {
        {
            // element k of row r goes to rows[r LP + ph(k)], copied
            // asynchronously so that all of the CTA's loads are in flight
            const int s = A.src.elem_stride;
            for (int r = 0; r < nrows; ++r) {
                const T* x = row_ptr(r);
                V* d = rows + (size_t)r * LP;
                for (int k = tid; k < L; k += NT) {
                    if (!STRIDED) {
                        cp_async<sizeof(V)>(d + ph<T>(k), reinterpret_cast<const V*>(x) + k);
                    } else {
                        cp_async<sizeof(T)>(&d[ph<T>(k)].x, x + (long long)(2 * k) * s);
                        cp_async<sizeof(T)>(&d[ph<T>(k)].y, x + (long long)(2 * k + 1) * s);
                    }
                }
            }
            load_twiddles_async(tws, A.twp,
                                LT > 0 ? FacOf<LT, sizeof(T) == 8>::v.twtotal : A.shape.twtotal);
            cp_async_wait_all();
        }
        __syncthreads();
        run_passes<T, LT>(rows, nrows, LP, A.shape, tws);
    }

    const int nout = (A.N + 1) * nf;
    const T rs = A.rowscale ? (T)A.rowscale[jh] : (T)1;
    // column maxima of the output (real and imaginary part of each field),
    // gathered per thread while its field stays the same, then per CTA in
    // shared memory, then one global atomic per column and CTA
    const bool track = A.colmax != nullptr;
    unsigned* smax = reinterpret_cast<unsigned*>(
        tws + (LT > 0 ? LT : (LT == -2 ? A.shape.L : A.L)));
    if (track) {
        for (int e = tid; e < 2 * nf; e += NT) smax[e] = 0u;
        __syncthreads();
    }
    float mre = 0.f, mim = 0.f;
    int mcur = -1;
    auto flush = [&]() {
        if (mcur >= 0) {
            atomicMax(&smax[2 * mcur], __float_as_uint(mre));
            atomicMax(&smax[2 * mcur + 1], __float_as_uint(mim));
        }
    };
    auto record = [&](int fl, V os, V oa) {
        if (fl != mcur) {
            flush();
            mcur = fl;
            mre = mim = 0.f;
        }
        mre = fmaxf(mre, fmaxf(fabsf((float)os.x), fabsf((float)oa.x)));
        mim = fmaxf(mim, fmaxf(fabsf((float)os.y), fabsf((float)oa.y)));
    };
    // 2 X_m = (Z_m + conj Z_{L-m}) + W_I^m (-i)(Z_m - conj Z_{L-m})
    auto real_spec = [&](V zm, V zc, V wt) -> V {
        // s = zm + conj zc, d = zm - conj zc; s + wt (-i d), componentwise
        const T sx = zm.x + zc.x, sy = zm.y - zc.y;
        const T dx = zm.x - zc.x, dy = zm.y + zc.y;
        return K::make(sx + wt.x * dy + wt.y * dx, sy - wt.x * dx + wt.y * dy);
    };
    // output scales, converted once (FP64 conversions use the narrow FP64 pipe)
    const T sc0 = (T)0.5 * rs * (T)A.mscale0, sc1 = (T)0.5 * rs * (T)A.mscale1;
    // two outputs (m, fl) per iteration, idx and idx + NT, with all shared-
    // memory reads of both issued before any arithmetic.  A reduced-grid row
    // of half-length L carries the wavenumbers up to min(N, L - 1); those
    // above are written as zeros (computed at the clamped wavenumber, then
    // discarded).  The loop is compiled twice, with and without that clamp.
    const int kmax = A.rowoff ? min(A.N, L - 1) : A.N;
    auto out_loop = [&](auto rag) {
        constexpr bool RAG = decltype(rag)::value;
        auto clampk = [&](int m) -> int {
            if constexpr (RAG)
                return min(m, kmax);
            else
                return m;
        };
        Walk2 wa(tid, nf), wb(tid + NT, nf);
        for (; wa.major * nf + wa.minor < nout; wa.next(), wa.next(), wb.next(), wb.next()) {
            const bool hb = wb.major * nf + wb.minor < nout;
            const int ma = wa.major, fa = wa.minor;
            const int mb = hb ? wb.major : ma, fb = hb ? wb.minor : fa;
            const int ra = clampk(ma), rb = clampk(mb);
            const int pma = ph<T>(rev_of<T, LT>(ra, A.rev));
            const int pca = ph<T>(rev_of<T, LT>(ra == 0 ? 0 : L - ra, A.rev));
            const int pmb = ph<T>(rev_of<T, LT>(rb, A.rev));
            const int pcb = ph<T>(rev_of<T, LT>(rb == 0 ? 0 : L - rb, A.rev));
            const V* na = rows + (size_t)fa * LP;
            const V* nb = rows + (size_t)fb * LP;
            V a_nm = na[pma], a_nc = na[pca], b_nm = nb[pmb], b_nc = nb[pcb];
            V a_sm = K::make((T)0, (T)0), a_sc = a_sm, b_sm = a_sm, b_sc = a_sm;
            if (!equator) {
                const V* sa = na + (size_t)nf * LP;
                const V* sb = nb + (size_t)nf * LP;
                a_sm = sa[pma];
                a_sc = sa[pca];
                b_sm = sb[pmb];
                b_sc = sb[pcb];
            }
            if constexpr (LT == -2) {   // Z_k = c_k conj(r_k)
                const V ca = A.chirp[ra], da = A.chirp[ra == 0 ? 0 : L - ra];
                const V cb = A.chirp[rb], db = A.chirp[rb == 0 ? 0 : L - rb];
                a_nm = K::mul(ca, K::conj(a_nm));
                a_nc = K::mul(da, K::conj(a_nc));
                a_sm = K::mul(ca, K::conj(a_sm));
                a_sc = K::mul(da, K::conj(a_sc));
                b_nm = K::mul(cb, K::conj(b_nm));
                b_nc = K::mul(db, K::conj(b_nc));
                b_sm = K::mul(cb, K::conj(b_sm));
                b_sc = K::mul(db, K::conj(b_sc));
            }
            const V wta = A.twpost[ra], wtb = A.twpost[rb];
            const T sca = ma == 0 ? sc0 : sc1;
            const T scb = mb == 0 ? sc0 : sc1;
            const V xan = real_spec(a_nm, a_nc, wta), xbn = real_spec(b_nm, b_nc, wtb);
            V Sa = xan, Aa = K::make((T)0, (T)0), Sb = xbn, Ab = Aa;
            if (!equator) {
                const V xas = real_spec(a_sm, a_sc, wta), xbs = real_spec(b_sm, b_sc, wtb);
                Sa = K::add(xan, xas);
                Aa = K::sub(xan, xas);
                Sb = K::add(xbn, xbs);
                Ab = K::sub(xbn, xbs);
            }
            V osa = K::scale(Sa, sca), oaa = K::scale(Aa, sca);
            if constexpr (RAG) {
                // rows shifted by half a spacing: X^m e^{-i pi m / I_j}
                if (A.shiftph) {
                    const V pa = A.shiftph[ra];
                    osa = K::mul(osa, pa);
                    oaa = K::mul(oaa, pa);
                }
            }
            if (ra != ma) osa = oaa = K::make((T)0, (T)0);
            const size_t basea = ((size_t)ma * 2 * A.Jh + jh) * A.F + f0 + fa;
            A.work[basea] = osa;
            A.work[basea + (size_t)A.Jh * A.F] = oaa;
            if (track) record(fa, osa, oaa);
            if (hb) {
                V osb = K::scale(Sb, scb), oab = K::scale(Ab, scb);
                if constexpr (RAG) {
                    if (A.shiftph) {
                        const V pb = A.shiftph[rb];
                        osb = K::mul(osb, pb);
                        oab = K::mul(oab, pb);
                    }
                }
                if (rb != mb) osb = oab = K::make((T)0, (T)0);
                const size_t baseb = ((size_t)mb * 2 * A.Jh + jh) * A.F + f0 + fb;
                A.work[baseb] = osb;
                A.work[baseb + (size_t)A.Jh * A.F] = oab;
                if (track) record(fb, osb, oab);
            }
        }
    };
    // The two-pass FP32 lengths L = Q x 32 on regular grids: each thread keeps
    // one field and walks the wavenumbers m = g, g + D, ... (D = NT / nf
    // thread groups), with the digit-reversed positions tracked as the
    // mixed-radix digits of m (m = k1 + Q k2 sits at 32 k1 + k2, padded
    // 33 k1 + k2; L - m at the digits of its complement) and the workspace
    // address advanced by a constant, so the loop needs no division.
    // Consecutive threads write consecutive fields of one m, as above.
    auto out_walk = [&]() {
        constexpr FftShape FS = FacOf<(LT > 0 ? LT : 64), false>::v;
        constexpr int Q = FS.radix[0];
        const int D = NT / nf;
        const int g = tid / nf, fl = tid - g * nf;
        if (g >= D) return;
        const V* zn = rows + (size_t)fl * LP;
        const V* zs = zn + (size_t)nf * LP;
        int k1 = g % Q, k2 = g / Q;
        const int d1 = D % Q, d2 = D / Q;
        V* wp = A.work + ((size_t)g * 2 * A.Jh + jh) * A.F + f0 + fl;
        const size_t wstep = (size_t)D * 2 * A.Jh * A.F;
        const size_t astep = (size_t)A.Jh * A.F;
        for (int m = g; m <= A.N; m += D) {
            const int c1 = k1 == 0 ? 0 : Q - k1;
            const int c2 = k1 == 0 ? ((32 - k2) & 31) : 31 - k2;
            const int pm = 33 * k1 + k2, pc = 33 * c1 + c2;
            const V wt = A.twpost[m];
            const V xn = real_spec(zn[pm], zn[pc], wt);
            V S = xn, Aq = K::make((T)0, (T)0);
            if (!equator) {
                const V xs = real_spec(zs[pm], zs[pc], wt);
                S = K::add(xn, xs);
                Aq = K::sub(xn, xs);
            }
            const T sc = m == 0 ? sc0 : sc1;
            const V os = K::scale(S, sc), oa = K::scale(Aq, sc);
            wp[0] = os;
            wp[astep] = oa;
            if (track) record(fl, os, oa);
            wp += wstep;
            k1 += d1;
            k2 += d2;
            if (k1 >= Q) {
                k1 -= Q;
                ++k2;
            }
        }
    };
    if constexpr (first_pass_from_global<T, LT>()) {
        if (!A.rowoff)
            out_walk();
        else
            out_loop(std::true_type{});
    } else {
        if (LT <= 0 || A.rowoff)
            out_loop(std::true_type{});
        else
            out_loop(std::false_type{});
    }
    if (track) {
        flush();
        __syncthreads();
        for (int e = tid; e < 2 * nf; e += NT) atomicMax(&A.colmax[2 * f0 + e], smax[e]);
    }
}

template <typename T, int LT, bool STRIDED>
__global__ void __launch_bounds__(NT, LT == -3 ? 3 : sizeof(T) == 4 ? 2 : 1)
    fft_forward_kernel(const __grid_constant__ FwdArgs<T> A) {
    begin_fft(A.follow);
    fwd_body<T, LT, STRIDED>(A, blockIdx.x, A.jh_list ? A.jh_list[blockIdx.y] : blockIdx.y);
    end_fft();
}

// PLAIN: the grid is only written (A.accumulate == 0).
template <typename T, int LT, bool PLAIN = false>
__device__ __forceinline__ void inv_body(const InvArgs<T>& A, int fg, int jh) {
    using V = typename Vec2<T>::type;
    using K = C2<T>;
    const int L = LT > 0 ? LT : A.L;
    const int LP = LT == -2 ? row_pitch<T>(A.shape.L) : A.LP;
    V* rows = reinterpret_cast<V*>(fft_smem_raw);
    V* tws = rows + (size_t)2 * A.G * LP;
    const int f0 = fg * A.G;
    const int nf = min(A.G, A.F - f0);
    const bool equator = (jh == A.Jh - 1);
    const int nrows = equator ? nf : 2 * nf;
    const int tid = threadIdx.x;
    const int half = L / 2;
    // Loads whose values are needed only after the copies below (the row
    // scale and, for compile-time lengths, the real-spectrum twiddles of the
    // thread's packing frequencies q and L - q), issued first so that their
    // latency hides behind the copies.
    const T rs = A.rowscale ? (T)A.rowscale[jh] : (T)1;
    constexpr int NQ = LT > 0 ? (LT / 2 + NT) / NT : 1;
    V twq[NQ], twc[NQ];
    if constexpr (LT > 0) {
#pragma unroll
        for (int i = 0; i < NQ; ++i) {
            const int q = tid + i * NT;
            if (q <= half) {
                twq[i] = A.twpost[q];
                twc[i] = A.twpost[q == 0 ? 0 : L - q];
            }
        }
    }

    load_twiddles(tws, A.twp, LT > 0 ? FacOf<LT, sizeof(T) == 8>::v.twtotal : A.shape.twtotal);
    // unfold S/A into the two hemispheres' zonal spectra Y_m, m <= N
    // (S lands in the northern row, A in the southern one, copied
    // asynchronously; then both hemispheres are formed in place)
    // a reduced-grid row of half-length L carries the wavenumbers up to
    // min(N, L - 1) (Y_m = 0 above)
    const int kmax = A.rowoff ? min(A.N, L - 1) : A.N;
    if constexpr (LT == -2) {   // zero padding of the convolution
        for (int r = 0; r < nrows; ++r)
            for (int n = L + tid; n < A.shape.L; n += NT)
                rows[(size_t)r * LP + ph<T>(n)] = K::make((T)0, (T)0);
    }
    const int nin = (kmax + 1) * nf;
    for (Walk2 w(tid, nf); w.major * nf + w.minor < nin; w.next()) {
        const int m = w.major, fl = w.minor;
        const size_t base = ((size_t)m * 2 * A.Jh + jh) * A.F + f0 + fl;
        cp_async<sizeof(V)>(rows + (size_t)fl * LP + ph<T>(m), A.work + base);
        if (!equator)
            cp_async<sizeof(V)>(rows + (size_t)(nf + fl) * LP + ph<T>(m),
                                A.work + base + (size_t)A.Jh * A.F);
    }
    cp_async_wait_all();
    __syncthreads();
    // One thread owns frequencies (q, L-q) of all fields in both hemispheres
    // Y_m = fac (S_m +- A_m) (Y_0 real, Y_m = 0 for m > kmax; stale slots
    // beyond kmax are never read), then the Hermitian packing
    //   Z_q = (Y_q + conj Y_{L-q}) + i conj(W_I^q) (Y_q - conj Y_{L-q}),
    // stored as conj(Z) in place.
    const T mf1 = (T)A.mfactor1;
    auto pack = [&](V y, V yc, V wv) -> V {
        return K::conj(K::add(K::add(y, K::conj(yc)),
                              K::mul_pi(K::mul(wv, K::sub(y, K::conj(yc))))));
    };
    // frequencies q and L - q with the twiddles W_I^q and W_I^{L-q}
    auto pack_q = [&](int q, V tq, V tc) {
        const int qc = L - q;   // >= q, as q <= L/2
        const int pq = ph<T>(q), pc = ph<T>(qc);
        const bool hq = q <= kmax, hc = q != 0 && qc <= kmax;
        const bool pair = q != 0 && q != qc;
        const T fq = q == 0 ? (T)1 : mf1, fc = mf1;
        const V wq = K::conj(tq);
        const V wc = pair ? K::conj(tc) : wq;
        const V zero = K::make((T)0, (T)0);
        // Bluestein rows: times the chirp
        const V hq_c = LT == -2 ? A.chirp[q] : zero, hc_c = LT == -2 && pair ? A.chirp[qc] : zero;
        auto chirped = [&](V z, V c) -> V { return LT == -2 ? K::mul(z, c) : z; };
        for (int fl = 0; fl < nf; ++fl) {
            V* zn = rows + (size_t)fl * LP;
            V* zs = rows + (size_t)(nf + fl) * LP;
            // S and A at frequencies q and L - q, each read once (zero above
            // kmax; Y_L = 0 for q = 0)
            V Sq = hq ? zn[pq] : zero;
            V Aq = (hq && !equator) ? zs[pq] : zero;
            V Sc = hc ? zn[pc] : zero;
            V Ac = (hc && !equator) ? zs[pc] : zero;
            if (A.shiftph) {
                // rows shifted by half a spacing: Y^m e^{+i pi m / I_j}
                const V cq = K::conj(A.shiftph[q]);
                Sq = K::mul(Sq, cq);
                Aq = K::mul(Aq, cq);
                if (hc) {
                    const V cc = K::conj(A.shiftph[qc]);
                    Sc = K::mul(Sc, cc);
                    Ac = K::mul(Ac, cc);
                }
            }
            V ynq = K::scale(K::add(Sq, Aq), fq), ysq = K::scale(K::sub(Sq, Aq), fq);
            if (q == 0) ynq.y = ysq.y = (T)0;
            const V ync = K::scale(K::add(Sc, Ac), fc), ysc = K::scale(K::sub(Sc, Ac), fc);
            zn[pq] = chirped(pack(ynq, ync, wq), hq_c);
            if (!equator) zs[pq] = chirped(pack(ysq, ysc, wq), hq_c);
            if (pair) {
                zn[pc] = chirped(pack(ync, ynq, wc), hc_c);
                if (!equator) zs[pc] = chirped(pack(ysc, ysq, wc), hc_c);
            }
        }
    };
    // When the spectrum stops below L/2 (kmax < L/2, i.e. I > 4 kmax, true of
    // every grid with I = 4 (N+1)), Y vanishes at L - q for all q <= L/2, so
    // each packed value depends on one Y:
    //   conj Z_q     = conj(Y_q) (1 - i W_I^q),
    //   conj Z_{L-q} = Y_q (1 + i W_I^{L-q}),
    // with the m >= 1 factor folded into the two constants, and both
    // hemispheres' Y = S +- A formed once per field.
    auto pack_q_short = [&](int q, V tq, V tc) {
        const int qc = L - q;
        const int pq = ph<T>(q), pc = ph<T>(qc);
        const bool pair = q != 0 && q != qc;
        const V zero = K::make((T)0, (T)0);
        const T fq = q == 0 ? (T)1 : mf1;
        V al = K::make(fq * ((T)1 + tq.y), -fq * tq.x);    // f (1 - i W^q)
        V be = K::make(mf1 * ((T)1 - tc.y), mf1 * tc.x);   // f (1 + i W^{L-q})
        if constexpr (LT == -2) {   // times the chirp
            al = K::mul(al, A.chirp[q]);
            if (pair) be = K::mul(be, A.chirp[qc]);
        }
        if (q > kmax) {
            for (int fl = 0; fl < nf; ++fl) {
                V* zn = rows + (size_t)fl * LP;
                V* zs = rows + (size_t)(nf + fl) * LP;
                zn[pq] = zero;
                if (!equator) zs[pq] = zero;
                if (pair) {
                    zn[pc] = zero;
                    if (!equator) zs[pc] = zero;
                }
            }
            return;
        }
        const V cs = A.shiftph ? K::conj(A.shiftph[q]) : K::make((T)1, (T)0);
        for (int fl = 0; fl < nf; ++fl) {
            V* zn = rows + (size_t)fl * LP;
            V* zs = rows + (size_t)(nf + fl) * LP;
            V Sq = zn[pq];
            V Aq = equator ? zero : zs[pq];
            if (A.shiftph) {
                Sq = K::mul(Sq, cs);
                Aq = K::mul(Aq, cs);
            }
            V yn = K::add(Sq, Aq), ys = K::sub(Sq, Aq);
            if (q == 0) yn.y = ys.y = (T)0;
            zn[pq] = K::mul(K::conj(yn), al);
            if (!equator) zs[pq] = K::mul(K::conj(ys), al);
            if (pair) {
                zn[pc] = K::mul(yn, be);
                if (!equator) zs[pc] = K::mul(ys, be);
            }
        }
    };
    const bool short_spec = 2 * kmax < L;
    if constexpr (LT > 0) {
        if (short_spec) {
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const int q = tid + i * NT;
                if (q <= half) pack_q_short(q, twq[i], twc[i]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < NQ; ++i) {
                const int q = tid + i * NT;
                if (q <= half) pack_q(q, twq[i], twc[i]);
            }
        }
    } else {
        for (int q = tid; q <= half; q += NT) {
            if (short_spec)
                pack_q_short(q, A.twpost[q], A.twpost[q == 0 ? 0 : L - q]);
            else
                pack_q(q, A.twpost[q], A.twpost[q == 0 ? 0 : L - q]);
        }
    }
    __syncthreads();
    if constexpr (inverse_stores_from_last_pass<T, LT>()) {
        if (PLAIN || A.accumulate == 0) {
            constexpr FftShape FS = FacOf<LT, false>::v;
            constexpr int R = FS.radix[1];   // 32 = the padding period: one padded
            constexpr int Q = FS.radix[0];   // index per butterfly
            passes_fixed<T, LT, 0, 1>(rows, nrows, LP, tws);
            const V sgn = K::make(rs, -rs);   // x = conj(z) rs
            constexpr int UNROLL = PLAIN ? 2 : 1;
#pragma unroll UNROLL
            for (int idx = tid; idx < nrows * Q; idx += NT) {
                const int r = idx / Q, b = idx - r * Q;
                const int f = f0 + (r < nf ? r : r - nf);
                const int j = (r < nf) ? jh : (A.J - 1 - jh);
                const long long off = A.rowoff ? (long long)f * A.fstride + A.rowoff[j]
                                               : ((long long)f * A.J + j) * A.I;
                V* xv = reinterpret_cast<V*>(A.grid + off) + b;
                const V* zb = rows + (size_t)r * LP + ph<T>(b * R);
                V a[R];
#pragma unroll
                for (int t = 0; t < R; ++t) a[t] = zb[t];
                Dft<T, R>::run(a);
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1)
                    xv[k1 * Q] = mul_f32x2(a[Dft<T, R>::pos(k1)], sgn);
            }
            return;
        }
        // onto the grid, or the products: the grid's values are read as well,
        // in row order after the last pass (below).  Read from the last
        // pass's registers, 64 bytes a row and warp at a time, the products
        // took 1340 us for Tc479 x 64, now 450.
    }
    if ((LT == -1 || LT == -3) && sizeof(T) == 4 && A.accumulate == 0 && A.shape.npass > 0) {
        // the last pass (span 1) straight to the grid rows, as above: the
        // butterfly of the digits k of the passes before it holds the
        // frequencies f + (L / R) k1, f = k_0 + r_0 (k_1 + r_1 (...)), so
        // lanes of consecutive f store consecutive values
        const int np = A.shape.npass;
        passes_runtime<T, LT == -1>(rows, nrows, LP, A.shape, 0, np - 1, tws);
        const V sgn = K::make(rs, -rs);   // x = conj(z) rs
        with_radix<T, LT == -1>(A.shape.radix[np - 1], [&](auto rc) {
            constexpr int R = decltype(rc)::value;
            const int nb = L / R;
            for (int idx = tid; idx < nrows * nb; idx += NT) {
                const int r = idx / nb, fb = idx - r * nb;
                int pos = 0, k = fb;
                for (int p = 0; p + 1 < np; ++p) {
                    const int kn = k / A.shape.radix[p];
                    pos += (k - kn * A.shape.radix[p]) * A.shape.span[p];
                    k = kn;
                }
                const int f = f0 + (r < nf ? r : r - nf);
                const int j = (r < nf) ? jh : (A.J - 1 - jh);
                const long long off = A.rowoff ? (long long)f * A.fstride + A.rowoff[j]
                                               : ((long long)f * A.J + j) * A.I;
                V* xv = reinterpret_cast<V*>(A.grid + off) + fb;
                const V* zb = rows + (size_t)r * LP;
                V a[R];
#pragma unroll
                for (int t = 0; t < R; ++t) a[t] = zb[ph<T>(pos + t)];
                Dft<T, R>::run(a);
#pragma unroll
                for (int k1 = 0; k1 < R; ++k1) {
                    const V y = a[Dft<T, R>::pos(k1)];
                    xv[k1 * nb] = K::make(y.x * sgn.x, y.y * sgn.y);
                }
            }
        });
        return;
    }
    if constexpr (LT == -2) {
        bluestein_rows<T>(rows, nrows, LP, A.shape, tws, A.dft);
    } else {
        run_passes<T, LT>(rows, nrows, LP, A.shape, tws);
    }

    // store of one synthesised pair of values y at xv[k] (x2: the second
    // grid of the products; g and h: the grids' values there, where read)
    auto put = [&](V* xv, V* x2, int k, V y, V g, V h) {
        if (A.accumulate == 1) {
            xv[k] = K::add(g, y);
        } else if (A.accumulate == 2) {
            const V uv = K::make(g.x * h.x, g.y * h.y);
            xv[k] = uv;
            x2[k] = K::make(uv.x * y.x, uv.y * y.y);
        } else {
            xv[k] = y;
        }
    };
    for (int r = 0; r < nrows; ++r) {
        const int f = f0 + (r < nf ? r : r - nf);
        const int j = (r < nf) ? jh : (A.J - 1 - jh);
        const long long off = A.rowoff ? (long long)f * A.fstride + A.rowoff[j]
                                       : ((long long)f * A.J + j) * A.I;
        V* xv = reinterpret_cast<V*>(A.grid + off);
        V* x2 = A.grid2 ? reinterpret_cast<V*>(A.grid2 + off) : nullptr;
        const V* z = rows + (size_t)r * LP;
        if constexpr (LT > 0) {
            // all of the thread's reads of the row first
            constexpr int NIT = (LT + NT - 1) / NT;
            V v[NIT], g[NIT], h[NIT];
#pragma unroll
            for (int i = 0; i < NIT; ++i) {
                const int k = tid + i * NT;
                if (LT % NT == 0 || k < LT) {
                    v[i] = z[ph<T>(rev_fixed<T, LT>(k))];
                    if (A.accumulate) g[i] = xv[k];
                    if (A.accumulate == 2) h[i] = x2[k];
                }
            }
#pragma unroll
            for (int i = 0; i < NIT; ++i) {
                const int k = tid + i * NT;
                if (LT % NT == 0 || k < LT)
                    put(xv, x2, k, K::make(v[i].x * rs, -v[i].y * rs), g[i], h[i]);
            }
        } else {
            constexpr int NB = 4;   // reads in flight per thread
            for (int k0 = tid; k0 < L; k0 += NB * NT) {
                V v[NB], g[NB], h[NB];
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    const int k = k0 + i * NT;
                    if (k >= L) continue;
                    v[i] = z[ph<T>(rev_of<T, LT>(k, A.rev))];
                    // Bluestein rows: DFT(conj Z)_k = c_k conj(r_k)
                    if constexpr (LT == -2) v[i] = K::mul(A.chirp[k], K::conj(v[i]));
                    if (A.accumulate) g[i] = xv[k];
                    if (A.accumulate == 2) h[i] = x2[k];
                }
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    const int k = k0 + i * NT;
                    if (k < L)
                        put(xv, x2, k, K::make(v[i].x * rs, -v[i].y * rs), g[i], h[i]);
                }
            }
        }
    }
}

template <typename T, int LT, bool PLAIN = false>
__global__ void __launch_bounds__(NT, LT == -3 ? 3 : sizeof(T) == 4 ? 2 : 1)
    fft_inverse_kernel(const __grid_constant__ InvArgs<T> A) {
    begin_fft(A.follow);
    inv_body<T, LT, PLAIN>(A, blockIdx.x, A.jh_list ? A.jh_list[blockIdx.y] : blockIdx.y);
    end_fft();
}

template <typename T>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 2 : 1)
    fft_forward_group_kernel(const __grid_constant__ FwdGroup<T> G) {
    begin_fft(G.follow);
    const int b = blockIdx.x;
    int p = 0;
    while (p + 1 < G.n && b >= G.cta_start[p + 1]) ++p;
    const int local = b - G.cta_start[p];
    const FwdArgs<T>& A = G.a[p];
    const int fg = local % G.nfg[p], jh = local / G.nfg[p];
    // the plan's half-length picks its compile-time body (one branch per CTA)
    switch (A.L) {
        case 64: fwd_body<T, 64, false>(A, fg, jh); break;
        case 128: fwd_body<T, 128, false>(A, fg, jh); break;
        case 256: fwd_body<T, 256, false>(A, fg, jh); break;
        case 320: fwd_body<T, 320, false>(A, fg, jh); break;
        case 512: fwd_body<T, 512, false>(A, fg, jh); break;
        case 640: fwd_body<T, 640, false>(A, fg, jh); break;
        case 1024: fwd_body<T, 1024, false>(A, fg, jh); break;
        case 1280: fwd_body<T, 1280, false>(A, fg, jh); break;
        default: fwd_body<T, -1, false>(A, fg, jh);
    }
}

template <typename T>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 2 : 1)
    fft_inverse_group_kernel(const __grid_constant__ InvGroup<T> G) {
    begin_fft(G.follow);
    const int b = blockIdx.x;
    int p = 0;
    while (p + 1 < G.n && b >= G.cta_start[p + 1]) ++p;
    const int local = b - G.cta_start[p];
    const InvArgs<T>& A = G.a[p];
    const int fg = local % G.nfg[p], jh = local / G.nfg[p];
    switch (A.L) {
        case 64: inv_body<T, 64>(A, fg, jh); break;
        case 128: inv_body<T, 128>(A, fg, jh); break;
        case 256: inv_body<T, 256>(A, fg, jh); break;
        case 320: inv_body<T, 320>(A, fg, jh); break;
        case 512: inv_body<T, 512>(A, fg, jh); break;
        case 640: inv_body<T, 640>(A, fg, jh); break;
        case 1024: inv_body<T, 1024>(A, fg, jh); break;
        case 1280: inv_body<T, 1280>(A, fg, jh); break;
        default: inv_body<T, -1>(A, fg, jh);
    }
}

template <typename T>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 2 : 1)
    fft_forward_ragged_kernel(const __grid_constant__ RaggedFwd<T> R) {
    begin_fft(R.follow);
    const int jh = R.a.jh_list[blockIdx.y];
    FwdArgs<T> A = R.a;
    apply_shape(A, R, jh);
    fwd_body<T, -1, false>(A, blockIdx.x, jh);
    end_fft();
}

template <typename T>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 2 : 1)
    fft_inverse_ragged_kernel(const __grid_constant__ RaggedInv<T> R) {
    begin_fft(R.follow);
    const int jh = R.a.jh_list[blockIdx.y];
    InvArgs<T> A = R.a;
    apply_shape(A, R, jh);
    inv_body<T, -1>(A, blockIdx.x, jh);
    end_fft();
}

// Rows whose half-length has a prime factor above 5: Bluestein's method.
template <typename T>
__global__ void __launch_bounds__(NT, 2)
    fft_forward_bluestein_kernel(const __grid_constant__ RaggedFwd<T> R) {
    begin_fft(R.follow);
    const int jh = R.a.jh_list[blockIdx.y];
    FwdArgs<T> A = R.a;
    apply_shape(A, R, jh);
    fwd_body<T, -2, false>(A, blockIdx.x, jh);
    end_fft();
}

template <typename T>
__global__ void __launch_bounds__(NT, 2)
    fft_inverse_bluestein_kernel(const __grid_constant__ RaggedInv<T> R) {
    begin_fft(R.follow);
    const int jh = R.a.jh_list[blockIdx.y];
    InvArgs<T> A = R.a;
    apply_shape(A, R, jh);
    inv_body<T, -2>(A, blockIdx.x, jh);
    end_fft();
}

// c_twf of this translation unit on the current device.
cudaError_t upload_twiddles() {
    float2 hf[kTwTotal];
    const long double pi = 3.14159265358979323846264338327950288L;
    for (int n : kComposite)
        for (int k = 0; k < n; ++k) {
            const long double ang = 2.0L * pi * (long double)k / (long double)n;
            const double c = (double)cosl(ang), sn = -(double)sinl(ang);
            hf[tw_offset(n) + k] = make_float2((float)c, (float)sn);
        }
    return cudaMemcpyToSymbol(c_twf, hf, sizeof(hf));
}

}  // namespace
}  // namespace sht
