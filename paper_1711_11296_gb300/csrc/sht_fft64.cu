// FP64 real FFTs along latitude circles in 64-bit fixed point, fused with the
// equatorial fold and the [m][parity][j][field] layout as in sht_fft.cu.
//
// The FP64 pipe of GB300 issues 2 operations per clock and SM, and a T639 row
// needs 53 000 of them: 32.7 / 34.3 ms (forward / inverse) for 256 fields,
// the pipe 99 % busy.  The integer pipes do 64 operations per clock and
// SM.  A row of FP64 values spans one scale (an FFT's rounding is relative to
// the row's magnitude whatever the format), so it can be transformed as
// 64-bit integers below that scale: an addition costs two integer
// instructions instead of 32 lanes' time on the FP64 pipe, a complex
// product 12 wide multiply-adds.
//
// Scale.  All rows of a field's latitude pair share the exponent e of their
// largest component; the integers are x 2^(SH - e), rounded.  A pass of radix
// R grows a modulus at most R-fold, and no partial sum exceeds the row's
// L1 norm, so after pass p the modulus is below
//   2^SH min(sqrt(2) R_0 ... R_p, L1 / 2^e) 2^-p,
// where every pass with twiddles halves its result (the product of a 64-bit
// integer with a twiddle in 2^-63 units, upper half).  SH is the largest
// that keeps this below 2^61.4, from the row's own maximum and L1 norm: 55
// for white noise at L = 1280, 53 for a constant row (where all that growth
// is in one value), 61 for a single point.
//
// Rounding (L = 1280, relative L2 error of the complex DFT, FP64 -> fixed
// point): white noise 2.9e-16 -> 2.2e-16, a zonal flow with 1.5 % noise 1.7e-16
// -> 0.8e-16 (the noise part alone 9.0e-16 -> 4.3e-16), a smooth row 1.8e-16
// -> 1.0e-16, a single point 1.5e-16 -> 1.0e-16.  That is relative to the
// latitude pair's largest value: what lies 2^-k below it keeps SH - k bits,
// where FP64 keeps 53 of each input (and of a sum, those of its largest term).
//
// Rows with an infinity or a NaN give NaN throughout (the FP64 transform's
// sums give NaN or an infinity).
//
// A CTA owns a latitude pair for G fields, as in sht_fft.cu: rows of
// 16-byte complex integers in the padded layout, radices 8 first, then 4, 2,
// 3, 5, each butterfly in registers; the first pass converts the FP64
// values as it reads them.  The kernel is bound by its phases' latency and
// by issue (T639: 14 500 instructions a row, half of the cycles issue one),
// so four CTAs share an SM: 64 registers, and the twiddle tables (20 KB at
// L = 1280) are read through L1 rather than copied to shared memory.
// Measured for 16 fields at T639, forward / inverse: 536 / 454 us with three
// CTAs and copied tables, 509 / 413 with four; 475 / 415 with the integer
// conversion.
#include "sht_fft_common.h"
#include "sht_internal.h"

namespace sht {
namespace {

constexpr int NT = kFftThreads;
using ll = long long;
using V = longlong2;

__device__ __forceinline__ V mk(ll x, ll y) { return make_longlong2(x, y); }
__device__ __forceinline__ V add(V a, V b) { return mk(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ V sub(V a, V b) { return mk(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ ll wide(int a, int b) { return (ll)a * b; }
// x = hi 2^32 + lo with lo in [-2^31, 2^31)
__device__ __forceinline__ int lo32(ll x) { return (int)x; }
__device__ __forceinline__ int hi32(ll x) {
    return (int)(x >> 32) + (int)((unsigned)x >> 31);
}

// z w / 2 for a twiddle w = {re hi, re lo, im hi, im lo} in 2^-63 units
// (|z| < 2^61.5).  Of the products with one low half only the upper words
// are formed (each rounded down: the four add a bias of -2 to the imaginary
// part, which is put back; in the real part it cancels), those of two low
// halves are left out: 0.6 in the last place rms.  64-bit sums of all cross
// products were more exact (0.3) but took 44 instructions instead of 30, and
// the input's rounding at 2^-SH is larger than either.
__device__ __forceinline__ V cmul63(V z, int4 w) {
    const int xl = lo32(z.x), xh = hi32(z.x), yl = lo32(z.y), yh = hi32(z.y);
    const int tr = __mulhi(xh, w.y) + __mulhi(xl, w.x) - (__mulhi(yh, w.w) + __mulhi(yl, w.z));
    const int ti =
        __mulhi(xh, w.w) + __mulhi(xl, w.z) + __mulhi(yh, w.y) + __mulhi(yl, w.x) + 2;
    return mk(wide(xh, w.x) - wide(yh, w.z) + (ll)tr, wide(xh, w.z) + wide(yh, w.x) + (ll)ti);
}

// x c / 2^64
template <ll CQ>
__device__ __forceinline__ ll mulc(ll x) {
    constexpr int cl = (int)CQ, ch = (int)((CQ - (ll)cl) >> 32);
    const int xl = lo32(x), xh = hi32(x);
    return wide(xh, ch) + (ll)(__mulhi(xh, cl) + __mulhi(xl, ch) + 1);
}

// constants c - 1 in 2^-64 units (c x = x + (c - 1) x)
constexpr ll kSqrtHalf = -5402926248376769404ll;    // sqrt(2)/2
constexpr ll kSin60 = -2471395088767036514ll;       // sqrt(3)/2
constexpr ll kSqrt5_4 = -8134700645620564469ll;     // sqrt(5)/4
constexpr ll kSin72 = -902847917979075853ll;        // sin(2 pi/5)
constexpr ll kSin36 = -7604019954369499282ll;       // sin(4 pi/5)

template <int R> struct Dft;

template <> struct Dft<2> {
    static __device__ __forceinline__ void run(V* a) {
        const V y = add(a[0], a[1]);
        a[1] = sub(a[0], a[1]);
        a[0] = y;
    }
};

template <> struct Dft<3> {
    static __device__ __forceinline__ void run(V* a) {
        const V t1 = add(a[1], a[2]), t2 = sub(a[1], a[2]);
        const ll hx = t2.x + mulc<kSin60>(t2.x), hy = t2.y + mulc<kSin60>(t2.y);
        const V m0 = mk(a[0].x - (t1.x >> 1), a[0].y - (t1.y >> 1));
        a[0] = add(a[0], t1);
        a[1] = mk(m0.x + hy, m0.y - hx);
        a[2] = mk(m0.x - hy, m0.y + hx);
    }
};

template <> struct Dft<4> {
    static __device__ __forceinline__ void run(V* a) {
        const V s02 = add(a[0], a[2]), d02 = sub(a[0], a[2]);
        const V s13 = add(a[1], a[3]), t = sub(a[1], a[3]);
        a[0] = add(s02, s13);
        a[2] = sub(s02, s13);
        a[1] = mk(d02.x + t.y, d02.y - t.x);
        a[3] = mk(d02.x - t.y, d02.y + t.x);
    }
};

template <> struct Dft<5> {
    static __device__ __forceinline__ void run(V* a) {
        // with cos(2 pi/5), cos(4 pi/5) = (-1 +- sqrt 5)/4
        const V b1 = add(a[1], a[4]), d1 = sub(a[1], a[4]);
        const V b2 = add(a[2], a[3]), d2 = sub(a[2], a[3]);
        const V b = add(b1, b2), c = sub(b1, b2);
        const V p0 = mk(a[0].x - (b.x >> 2), a[0].y - (b.y >> 2));
        const V pc = mk(c.x + mulc<kSqrt5_4>(c.x), c.y + mulc<kSqrt5_4>(c.y));
        a[0] = add(a[0], b);
        const V p1 = add(p0, pc), p2 = sub(p0, pc);
        // q1 = s1 d1 + s2 d2, q2 = s2 d1 - s1 d2
        auto q1 = [](ll u, ll v) { return u + v + mulc<kSin72>(u) + mulc<kSin36>(v); };
        auto q2 = [](ll u, ll v) { return u - v + mulc<kSin36>(u) - mulc<kSin72>(v); };
        const V e = mk(q1(d1.x, d2.x), q1(d1.y, d2.y)), f = mk(q2(d1.x, d2.x), q2(d1.y, d2.y));
        a[1] = mk(p1.x + e.y, p1.y - e.x);
        a[4] = mk(p1.x - e.y, p1.y + e.x);
        a[2] = mk(p2.x + f.y, p2.y - f.x);
        a[3] = mk(p2.x - f.y, p2.y + f.x);
    }
};

template <> struct Dft<8> {
    static __device__ __forceinline__ void run(V* a) {
        V e[4] = {a[0], a[2], a[4], a[6]};
        V o[4] = {a[1], a[3], a[5], a[7]};
        Dft<4>::run(e);
        Dft<4>::run(o);
        auto r = [](ll x) { return x + mulc<kSqrtHalf>(x); };
        const V o1 = mk(r(o[1].x + o[1].y), r(o[1].y - o[1].x));     // W8^1 o1
        const V o3 = mk(r(o[3].y - o[3].x), -r(o[3].x + o[3].y));    // W8^3 o3
        a[0] = add(e[0], o[0]);
        a[4] = sub(e[0], o[0]);
        a[1] = add(e[1], o1);
        a[5] = sub(e[1], o1);
        a[2] = mk(e[2].x + o[2].y, e[2].y - o[2].x);
        a[6] = mk(e[2].x - o[2].y, e[2].y + o[2].x);
        a[3] = add(e[3], o3);
        a[7] = sub(e[3], o3);
    }
};

// ---- FP64 <-> fixed point --------------------------------------------------

// Per field of the CTA: largest |component| (high word of its FP64 bits)
// and the warps' shares of the L1 norms of its two rows (added in a fixed
// order, so that the scale does not depend on timing) while they are
// gathered, then the exponent shift of the conversion and the factors of
// the way back.
struct Field {
    unsigned hmax;
    int shift;       // SH - e: integer = round(v 2^shift)
    double sc, sc2;  // integer -> FP64: times sc (times sc2 at the range's end)
    float l1[2][NT / 32];
    __device__ __forceinline__ float norm(int row) const {
        float x = 0.f;
#pragma unroll
        for (int w = 0; w < NT / 32; ++w) x += l1[row][w];
        return x;
    }
};
static_assert(sizeof(Field) <= kFxFieldBytes, "the launches reserve this much per field");

__device__ __forceinline__ unsigned hi_abs(double v) {
    return (unsigned)(__double_as_longlong(v) >> 32) & 0x7fffffffu;
}

// |v| truncated to 20 bits of mantissa as FP32, from its high word; below
// 2^-126 it reads as 0, above 2^128 wrongly (finish_field tells from the
// maximum).  Integer operations: a conversion would take the FP64 pipe.
__device__ __forceinline__ float abs_f32(unsigned h) {
    return __int_as_float(max((int)h - (896 << 20), 0) << 3);
}

// round(v 2^shift), |result| <= 2^61, shift <= 1082.  Integer operations: as a conversion on
// the FP64 pipe the first pass of the forward took 7 % longer.
__device__ __forceinline__ ll to_fx(double v, int shift) {
    const ll bits = __double_as_longlong(v);
    const int ex = (int)(bits >> 52) & 0x7ff;
    ll man = bits & 0xfffffffffffffll;
    if (ex) man |= 0x10000000000000ll;
    const int d = min(1083 - shift - max(ex, 1), 63);
    const ll t = (ll)(((unsigned long long)(man << 9) >> d) + 1) >> 1;
    return bits < 0 ? -t : t;
}

// SH and the scales of one field from its gathered maximum and L1 norm l1 (in
// units of 2^e: |v| < 2^e).  b(l1): largest bound of the modulus over the
// passes, in units of 2^SH; k: the transform's value is
// integer * 2^(e - SH + k), times f.
template <class Bound>
__device__ __forceinline__ void finish_field(Field& fd, float l1, Bound bound, double f) {
    const int E = (int)(fd.hmax >> 20);   // biased exponent field
    // (subnormals: below 2^(bits of the high word - 1042))
    const int e = E > 0 ? E - 1022 : 32 - __clz((int)fd.hmax) - 1042;
    // without a usable FP32 sum the maximum alone bounds the growth
    l1 = (E >= 940 && E <= 1140) ? l1 * 1.0001f * __int_as_float((127 - e) << 23)
                                 : __int_as_float(0x7f800000);
    int k;
    const float b = bound(l1, k);
    const int SH = min(61, (int)floorf(61.4f - log2f(b)));
    fd.shift = min(SH - e, 1082);   // as far as to_fx shifts
    const int p2 = k - fd.shift;
    const bool tiny = p2 < -900;   // 2^p2 would be subnormal
    // (zero rows give zeros, not the last place's rounding)
    fd.sc = E == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll)
            : fd.hmax == 0u ? 0.0
                            : ldexp(f, tiny ? p2 + 200 : p2);
    fd.sc2 = tiny ? 6.223015277861142e-61 : 1.0;   // 2^-200
}

__device__ __forceinline__ double from_fx(ll x, double sc, double sc2) {
    const double d = __ll2double_rn(x) * sc;
    return sc2 == 1.0 ? d : d * sc2;
}

// The same for a scale that is a power of two (|sc| in range, or NaN: the
// exponent is then not a plain one), by an integer addition to the exponent.
__device__ __forceinline__ double from_fx_pow2(ll x, int p2) {
    const double d = __ll2double_rn(x);
    return x == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (p2 << 20), __double2loint(d));
}

// ---- passes -------------------------------------------------------------------

// One butterfly of radix R over span M (M <= 0: run-time span Mr); FIRST reads
// FP64 values.  Results with twiddles (span > 1) are halved.
template <int R, int M, bool FIRST>
__device__ __forceinline__ void bfly(V* z, int at, int Mr, const int4* tw, int n1, int shift) {
    const int m = M > 0 ? M : Mr;
    V a[R];
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const int i = ph<double>(at + t * m);
        if constexpr (FIRST) {
            const double2 d = reinterpret_cast<const double2*>(z)[i];
            a[t] = mk(to_fx(d.x, shift), to_fx(d.y, shift));
        } else {
            a[t] = z[i];
        }
    }
    Dft<R>::run(a);
    if (M != 1 && m > 1) {
        a[0] = mk(a[0].x >> 1, a[0].y >> 1);
        if (n1 != 0) {
#pragma unroll
            for (int k1 = 1; k1 < R; ++k1) a[k1] = cmul63(a[k1], __ldg(tw + (k1 - 1) * m + n1));
        } else {
#pragma unroll
            for (int k1 = 1; k1 < R; ++k1) a[k1] = mk(a[k1].x >> 1, a[k1].y >> 1);
        }
    }
#pragma unroll
    for (int k1 = 0; k1 < R; ++k1) z[ph<double>(at + k1 * m)] = a[k1];
}

template <bool FIRST>
__device__ __forceinline__ void pass_rt(V* rows, int nrows, int nf, int LP, const FftShape& sh,
                                        int p, const int4* twp, const Field* fd) {
    const int r = sh.radix[p], M = sh.span[p], S = r * M, nb = sh.L / r;
    const int4* tw = twp + sh.twoff[p];
    for (int idx = threadIdx.x; idx < nrows * nb; idx += NT) {
        const int row = idx / nb, b = idx - row * nb;
        const int blk = b / M, n1 = b - blk * M;
        V* z = rows + (size_t)row * LP;
        const int at = blk * S + n1;
        const int shift = FIRST ? fd[row < nf ? row : row - nf].shift : 0;
        if (r == 8) bfly<8, 0, FIRST>(z, at, M, tw, n1, shift);
        else if (r == 4) bfly<4, 0, FIRST>(z, at, M, tw, n1, shift);
        else if (r == 2) bfly<2, 0, FIRST>(z, at, M, tw, n1, shift);
        else if (r == 5) bfly<5, 0, FIRST>(z, at, M, tw, n1, shift);
        else bfly<3, 0, FIRST>(z, at, M, tw, n1, shift);
    }
    __syncthreads();
}

template <int L, int P, bool CONV>
__device__ __forceinline__ void passes_ct(V* rows, int nrows, int nf, int LP, const int4* twp,
                                          const Field* fd) {
    constexpr FftShape F = FacOf<L, true>::v;
    if constexpr (P < F.npass) {
        constexpr int R = F.radix[P], M = F.span[P], S = R * M, NB = L / R;
        constexpr bool FIRST = CONV && P == 0;
        for (int idx = threadIdx.x; idx < nrows * NB; idx += NT) {
            const int row = idx / NB, b = idx - row * NB;
            const int blk = b / M, n1 = b - blk * M;
            const int shift = FIRST ? fd[row < nf ? row : row - nf].shift : 0;
            bfly<R, M, FIRST>(rows + (size_t)row * LP, blk * S + n1, M, twp + F.twoff[P], n1,
                              shift);
        }
        __syncthreads();
        passes_ct<L, P + 1, CONV>(rows, nrows, nf, LP, twp, fd);
    }
}

// In-place FFT of nrows padded rows; CONV: the rows hold FP64 values.
template <int LT, bool CONV>
__device__ __forceinline__ void passes(V* rows, int nrows, int nf, int LP, const FftShape& sh,
                                       const int4* twp, const Field* fd) {
    if constexpr (LT > 0) {
        passes_ct<LT, 0, CONV>(rows, nrows, nf, LP, twp, fd);
    } else {
        if (CONV && sh.npass == 0) {   // rows of one complex value
            for (int r = threadIdx.x; r < nrows; r += NT) {
                const double2 d = reinterpret_cast<const double2*>(rows)[(size_t)r * LP];
                const int shift = fd[r < nf ? r : r - nf].shift;
                rows[(size_t)r * LP] = mk(to_fx(d.x, shift), to_fx(d.y, shift));
            }
            __syncthreads();
        }
        for (int p = 0; p < sh.npass; ++p) {
            if (CONV && p == 0)
                pass_rt<true>(rows, nrows, nf, LP, sh, p, twp, fd);
            else
                pass_rt<false>(rows, nrows, nf, LP, sh, p, twp, fd);
        }
    }
}

// Largest modulus over the passes in units of 2^SH: inputs of modulus zmax and
// L1 norm l1; the last pass's result times `last`.  Also the number of
// halvings (passes with twiddles).
template <int LT>
__device__ __forceinline__ float pass_bound(const FftShape& sh, float zmax, float l1, float last,
                                            int& halvings) {
    auto run = [&](const FftShape& F) {
        float P = zmax, g = 1.f, b = fminf(zmax, l1);
        int h = 0;
#pragma unroll
        for (int p = 0; p < (LT > 0 ? FacOf<(LT > 0 ? LT : 2), true>::v.npass : F.npass); ++p) {
            P *= (float)F.radix[p];
            b = fmaxf(b, fminf(P, l1) * g);
            if (F.span[p] > 1) {
                g *= 0.5f;
                ++h;
            }
        }
        halvings = h;
        return fmaxf(b, fminf(P, l1) * g * last);
    };
    if constexpr (LT > 0) {
        constexpr FftShape F = FacOf<LT, true>::v;
        return run(F);
    } else {
        return run(sh);
    }
}

// Reduce a thread's share of one row into its field.  low: its values' low words,
// which tell the smallest subnormals (high word 0) from zeros.
__device__ __forceinline__ void gather_row(Field& fd, int row, unsigned hm, int low, float l1) {
    if (low != 0) hm = max(hm, 1u);
    hm = __reduce_max_sync(0xffffffffu, hm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&fd.hmax, hm);
        fd.l1[row][threadIdx.x >> 5] = l1;
    }
}

extern __shared__ __align__(16) unsigned char fx_smem[];

template <int LT, bool STRIDED>
__device__ __forceinline__ void fwd_body(const FwdArgs<double>& A, int fg, int jh) {
    const int L = LT > 0 ? LT : A.L;
    const int LP = A.LP;
    V* rows = reinterpret_cast<V*>(fx_smem);
    const double2* raw = reinterpret_cast<const double2*>(fx_smem);
    const int4* tws = reinterpret_cast<const int4*>(A.twp);
    Field* fd = reinterpret_cast<Field*>(rows + (size_t)2 * A.G * LP);
    const int f0 = fg * A.G;
    const int nf = min(A.G, A.F - f0);
    const bool equator = (jh == A.Jh - 1);
    const int nrows = equator ? nf : 2 * nf;
    const int tid = threadIdx.x;

    for (int f = tid; f < nf; f += NT) {
        fd[f].hmax = 0u;
        for (int w = 0; w < NT / 32; ++w) fd[f].l1[1][w] = 0.f;   // no southern Equator row
    }
    const int s = A.src.elem_stride;
    for (int r = 0; r < nrows; ++r) {
        const int f = f0 + (r < nf ? r : r - nf);
        const int j = (r < nf) ? jh : (A.J - 1 - jh);
        const double* x = A.grid + (long long)f * A.src.field_stride +
                          (A.rowoff ? A.rowoff[j]
                                    : A.src.row_offset + (long long)j * A.src.row_stride);
        double2* d = reinterpret_cast<double2*>(rows) + (size_t)r * LP;
        for (int k = tid; k < L; k += NT) {
            if (!STRIDED) {
                cp_async<16>(d + ph<double>(k), reinterpret_cast<const double2*>(x) + k);
            } else {
                cp_async<8>(&d[ph<double>(k)].x, x + (long long)(2 * k) * s);
                cp_async<8>(&d[ph<double>(k)].y, x + (long long)(2 * k + 1) * s);
            }
        }
    }
    cp_async_wait_all();
    __syncthreads();
    // the largest component of each field and the L1 norm of each row
    for (int r = 0; r < nrows; ++r) {
        unsigned hm = 0u;
        int low = 0;
        float l1 = 0.f;
        for (int k = tid; k < L; k += NT) {
            const double2 v = raw[(size_t)r * LP + ph<double>(k)];
            const unsigned hx = hi_abs(v.x), hy = hi_abs(v.y);
            hm = max(hm, max(hx, hy));
            low |= __double2loint(v.x) | __double2loint(v.y);
            l1 += abs_f32(hx) + abs_f32(hy);
        }
        gather_row(fd[r < nf ? r : r - nf], r < nf ? 0 : 1, hm, low, l1);
    }
    __syncthreads();
    if (tid < nf) {
        Field& q = fd[tid];
        finish_field(
            q, fmaxf(q.norm(0), q.norm(1)),
            [&](float l1, int& k) { return pass_bound<LT>(A.shape, 1.4142136f, l1, 2.f, k); },
            A.rowscale ? A.rowscale[jh] : 1.0);
    }
    __syncthreads();
    passes<LT, true>(rows, nrows, nf, LP, A.shape, tws, fd);

    // X_m = ((Z_m + conj Z_{L-m}) + W_I^m (-i)(Z_m - conj Z_{L-m})) / 2: the
    // product with W is halved by itself, the sum by a shift
    const int4* post = reinterpret_cast<const int4*>(A.twpost);
    auto real_spec = [&](V zm, V zc, int4 w, bool m0) -> V {
        const V u = mk(zm.y + zc.y, zc.x - zm.x);   // -i (zm - conj zc)
        const V t = m0 ? mk(u.x >> 1, u.y >> 1) : cmul63(u, w);
        return mk(((zm.x + zc.x) >> 1) + t.x, ((zm.y - zc.y) >> 1) + t.y);
    };
    const int kmax = A.rowoff ? min(A.N, L - 1) : A.N;
    const size_t astep = (size_t)A.Jh * A.F;
    for (Walk2 w(tid, nf); w.major <= A.N; w.next()) {
        const int m = w.major, fl = w.minor;
        double2 os = make_double2(0.0, 0.0), oa = os;
        if (m <= kmax) {
            const int pm = ph<double>(__ldg(A.rev + m));
            const int pc = ph<double>(__ldg(A.rev + (m == 0 ? 0 : L - m)));
            const int4 wt = post[m];
            const V* zn = rows + (size_t)fl * LP;
            const V xn = real_spec(zn[pm], zn[pc], wt, m == 0);
            V S = xn, D = mk(0, 0);
            if (!equator) {
                const V* zs = zn + (size_t)nf * LP;
                const V xs = real_spec(zs[pm], zs[pc], wt, m == 0);
                S = add(xn, xs);
                D = sub(xn, xs);
            }
            const double sc = fd[fl].sc * (m == 0 ? A.mscale0 : A.mscale1), sc2 = fd[fl].sc2;
            os = make_double2(from_fx(S.x, sc, sc2), from_fx(S.y, sc, sc2));
            oa = make_double2(from_fx(D.x, sc, sc2), from_fx(D.y, sc, sc2));
            if (A.shiftph) {
                // rows shifted by half a spacing: X^m e^{-i pi m / I_j}
                const double2 p = A.shiftph[m];
                os = make_double2(os.x * p.x - os.y * p.y, os.x * p.y + os.y * p.x);
                oa = make_double2(oa.x * p.x - oa.y * p.y, oa.x * p.y + oa.y * p.x);
            }
        }
        double2* wp = A.work + ((size_t)m * 2 * A.Jh + jh) * A.F + f0 + fl;
        wp[0] = os;
        wp[astep] = oa;
    }
}

template <int LT>
__device__ __forceinline__ void inv_body(const InvArgs<double>& A, int fg, int jh) {
    const int L = LT > 0 ? LT : A.L;
    const int LP = A.LP;
    V* rows = reinterpret_cast<V*>(fx_smem);
    const double2* raw = reinterpret_cast<const double2*>(fx_smem);
    const int4* tws = reinterpret_cast<const int4*>(A.twp);
    Field* fd = reinterpret_cast<Field*>(rows + (size_t)2 * A.G * LP);
    const int f0 = fg * A.G;
    const int nf = min(A.G, A.F - f0);
    const bool equator = (jh == A.Jh - 1);
    const int nrows = equator ? nf : 2 * nf;
    const int tid = threadIdx.x;
    for (int f = tid; f < nf; f += NT) {
        fd[f].hmax = 0u;
        for (int w = 0; w < NT / 32; ++w) fd[f].l1[1][w] = 0.f;   // no southern Equator row
    }
    // S lands in the northern row, A in the southern one; a reduced-grid row
    // carries the wavenumbers up to min(N, L - 1)
    const int kmax = A.rowoff ? min(A.N, L - 1) : A.N;
    for (Walk2 w(tid, nf); w.major <= kmax; w.next()) {
        const int m = w.major, fl = w.minor;
        const double2* src = A.work + ((size_t)m * 2 * A.Jh + jh) * A.F + f0 + fl;
        double2* d = reinterpret_cast<double2*>(rows) + (size_t)fl * LP + ph<double>(m);
        cp_async<16>(d, src);
        if (!equator) cp_async<16>(d + (size_t)nf * LP, src + (size_t)A.Jh * A.F);
    }
    cp_async_wait_all();
    __syncthreads();
    // the largest component of S and A of each field and their L1 norms (Im
    // at m = 0 is not an input; Re there counts twice, as Y_0 may)
    for (int r = 0; r < nrows; ++r) {
        unsigned hm = 0u;
        int low = 0;
        float l1 = 0.f;
        for (int k = tid; k <= kmax; k += NT) {
            const double2 v = raw[(size_t)r * LP + ph<double>(k)];
            const double y = k == 0 ? v.x : v.y;
            const unsigned hx = hi_abs(v.x), hy = hi_abs(y);
            hm = max(hm, max(hx, hy));
            low |= __double2loint(v.x) | __double2loint(y);
            l1 += abs_f32(hx) + abs_f32(hy);
        }
        gather_row(fd[r < nf ? r : r - nf], r < nf ? 0 : 1, hm, low, l1);
    }
    __syncthreads();
    // The factor of the m >= 1 terms (1, or 1/2 for an adjoint) goes into the
    // scale, its inverse into Y_0.
    const int y0_shift = A.mfactor1 == 0.5 ? 1 : 0;
    if (tid < nf) {
        Field& q = fd[tid];
        // packed values: |Z_q| / 2 <= |Y_q| + |Y_{L-q}|, |Y| <= |S| + |A|; the
        // phase of a shifted row may raise a component by sqrt(2)
        if (A.shiftph && q.hmax < 0x7fe00000u) q.hmax += min(q.hmax, 0x100000u);
        finish_field(
            q, q.norm(0) + q.norm(1),
            [&](float l1, int& k) {
                // (two outputs per input: the L1 norm of the packed values)
                const float b = pass_bound<LT>(A.shape, 5.656855f, 2.f * l1, 1.f, k);
                ++k;
                return b;
            },
            A.mfactor1 * (A.rowscale ? A.rowscale[jh] : 1.0));
    }
    __syncthreads();
    // One thread owns frequencies q and L - q of all fields and both
    // hemispheres.  With a = Y_q + conj Y_{L-q}, b = Y_q - conj Y_{L-q} and
    // t = -i W_I^q conj(b):
    //   conj Z_q = conj a + t,  conj Z_{L-q} = conj(conj a - t),
    // both halved (the product with W is halved by itself).
    const int4* post = reinterpret_cast<const int4*>(A.twpost);
    for (int q = tid; q <= L / 2; q += NT) {
        const int qc = L - q;
        const int pq = ph<double>(q), pc = ph<double>(qc);
        const bool hq = q <= kmax, hc = q != 0 && qc <= kmax, pair = q != 0 && q != qc;
        const int4 wt = post[q < L ? q : 0];
        for (int fl = 0; fl < nf; ++fl) {
            V* zn = rows + (size_t)fl * LP;
            V* zs = zn + (size_t)nf * LP;
            const int shift = fd[fl].shift;
            auto get = [&](const V* z, int pos, int k) -> V {
                double2 d = reinterpret_cast<const double2*>(z)[pos];
                if (A.shiftph) {
                    // rows shifted by half a spacing: Y^m e^{+i pi m / I_j}
                    const double2 p = A.shiftph[k];
                    if (k == 0) d.y = 0.0;
                    d = make_double2(d.x * p.x + d.y * p.y, d.y * p.x - d.x * p.y);
                }
                return mk(to_fx(d.x, shift), to_fx(d.y, shift));
            };
            const V zero = mk(0, 0);
            const V Sq = hq ? get(zn, pq, q) : zero, Aq = hq && !equator ? get(zs, pq, q) : zero;
            const V Sc = hc ? get(zn, pc, qc) : zero, Ac = hc && !equator ? get(zs, pc, qc) : zero;
            auto put = [&](V* z, V y, V yc) {
                if (q == 0) y = mk(y.x << y0_shift, 0);
                // conj a, and -i conj b: (b.x - i b.y)(-i) = -b.y - i b.x
                const V ca = mk(y.x + yc.x, yc.y - y.y);
                const V u = mk(-(y.y + yc.y), yc.x - y.x);
                const V t = q == 0 ? mk(u.x >> 1, u.y >> 1) : cmul63(u, wt);
                const ll hx = ca.x >> 1, hy = ca.y >> 1;
                z[pq] = mk(hx + t.x, hy + t.y);
                if (pair) z[pc] = mk(hx - t.x, t.y - hy);
            };
            put(zn, add(Sq, Aq), add(Sc, Ac));
            if (!equator) put(zs, sub(Sq, Aq), sub(Sc, Ac));
        }
    }
    __syncthreads();
    passes<LT, false>(rows, nrows, nf, LP, A.shape, tws, fd);

    for (int r = 0; r < nrows; ++r) {
        const int fl = r < nf ? r : r - nf, f = f0 + fl;
        const int j = (r < nf) ? jh : (A.J - 1 - jh);
        const long long off = A.rowoff ? (long long)f * A.fstride + A.rowoff[j]
                                       : ((long long)f * A.J + j) * A.I;
        double2* xv = reinterpret_cast<double2*>(A.grid + off);
        double2* x2 = A.grid2 ? reinterpret_cast<double2*>(A.grid2 + off) : nullptr;
        const V* z = rows + (size_t)r * LP;
        const double sc = fd[fl].sc, sc2 = fd[fl].sc2;
        // without row weights the scale is a power of two (exponent p2, far
        // inside the range unless the field is at its ends)
        const int p2 = ((__double2hiint(sc) >> 20) & 0x7ff) - 1023;
        const bool pow2 = A.rowscale == nullptr && sc2 == 1.0 && p2 > -900 && p2 < 900;
        for (int k = tid; k < L; k += NT) {
            const V v = z[ph<double>(__ldg(A.rev + k))];
            double2 y;
            if (pow2)
                y = make_double2(from_fx_pow2(v.x, p2), from_fx_pow2(-v.y, p2));
            else
                y = make_double2(from_fx(v.x, sc, sc2), from_fx(-v.y, sc, sc2));
            if (A.accumulate == 1) {
                const double2 g = xv[k];
                y = make_double2(g.x + y.x, g.y + y.y);
            } else if (A.accumulate == 2) {
                const double2 g = xv[k], h = x2[k];
                const double2 uv = make_double2(g.x * h.x, g.y * h.y);
                x2[k] = make_double2(uv.x * y.x, uv.y * y.y);
                y = uv;
            }
            xv[k] = y;
        }
    }
}

template <int LT, bool STRIDED>
__global__ void __launch_bounds__(NT, 4)
    fx_forward_kernel(const __grid_constant__ FwdArgs<double> A) {
    begin_fft(A.follow);
    fwd_body<LT, STRIDED>(A, blockIdx.x, A.jh_list ? A.jh_list[blockIdx.y] : blockIdx.y);
    end_fft();
}

template <int LT>
__global__ void __launch_bounds__(NT, 4)
    fx_inverse_kernel(const __grid_constant__ InvArgs<double> A) {
    begin_fft(A.follow);
    inv_body<LT>(A, blockIdx.x, A.jh_list ? A.jh_list[blockIdx.y] : blockIdx.y);
    end_fft();
}

__global__ void __launch_bounds__(NT, 4)
    fx_forward_ragged_kernel(const __grid_constant__ RaggedFwd<double> R) {
    begin_fft(R.follow);
    const int jh = R.a.jh_list[blockIdx.y];
    FwdArgs<double> A = R.a;
    apply_shape(A, R, jh);
    fwd_body<-1, false>(A, blockIdx.x, jh);
    end_fft();
}

__global__ void __launch_bounds__(NT, 4)
    fx_inverse_ragged_kernel(const __grid_constant__ RaggedInv<double> R) {
    begin_fft(R.follow);
    const int jh = R.a.jh_list[blockIdx.y];
    InvArgs<double> A = R.a;
    apply_shape(A, R, jh);
    inv_body<-1>(A, blockIdx.x, jh);
    end_fft();
}

#define SHT_FX_BODY(L, CALL)               \
    switch (L) {                           \
        case 64: CALL(64); break;          \
        case 128: CALL(128); break;        \
        case 256: CALL(256); break;        \
        case 320: CALL(320); break;        \
        case 512: CALL(512); break;        \
        case 640: CALL(640); break;        \
        case 1024: CALL(1024); break;      \
        case 1280: CALL(1280); break;      \
        default: CALL(-1);                 \
    }

// the plan's half-length picks its compile-time body (one branch per CTA)
__global__ void __launch_bounds__(NT, 4)
    fx_forward_group_kernel(const __grid_constant__ FwdGroup<double> G) {
    begin_fft(G.follow);
    const int b = blockIdx.x;
    int p = 0;
    while (p + 1 < G.n && b >= G.cta_start[p + 1]) ++p;
    const int local = b - G.cta_start[p];
    const FwdArgs<double>& A = G.a[p];
    const int fg = local % G.nfg[p], jh = local / G.nfg[p];
#define SHT_CALL(LV) fwd_body<LV, false>(A, fg, jh)
    SHT_FX_BODY(A.L, SHT_CALL)
#undef SHT_CALL
}

__global__ void __launch_bounds__(NT, 4)
    fx_inverse_group_kernel(const __grid_constant__ InvGroup<double> G) {
    begin_fft(G.follow);
    const int b = blockIdx.x;
    int p = 0;
    while (p + 1 < G.n && b >= G.cta_start[p + 1]) ++p;
    const int local = b - G.cta_start[p];
    const InvArgs<double>& A = G.a[p];
    const int fg = local % G.nfg[p], jh = local / G.nfg[p];
#define SHT_CALL(LV) inv_body<LV>(A, fg, jh)
    SHT_FX_BODY(A.L, SHT_CALL)
#undef SHT_CALL
}

// FP64 twiddles to 2^-63 units, in place: each component as hi 2^32 + lo with
// lo in [-2^31, 2^31).  The components of the tables' used entries are
// below 1 (-1 fits): entry 0 of the real-spectrum table and n1 = 0 of a
// pass, where W = 1, are not read.
__global__ void fixed_twiddle_kernel(double2* t, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    auto conv = [](double v, int& h, int& l) {
        const ll q = v >= 1.0 ? 0x7fffffffffffffffll : __double2ll_rn(v * 9223372036854775808.0);
        l = (int)q;
        h = (int)((q - (ll)l) >> 32);
    };
    const double2 v = t[i];
    int4 w;
    conv(v.x, w.x, w.y);
    conv(v.y, w.z, w.w);
    reinterpret_cast<int4*>(t)[i] = w;
}

}  // namespace

cudaError_t launch_fixed_twiddles(void* table, int n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    fixed_twiddle_kernel<<<(n + 127) / 128, 128, 0, s>>>(static_cast<double2*>(table), n);
    return cudaGetLastError();
}

cudaError_t fx_forward(const FwdArgs<double>& A, bool strided, dim3 grid, size_t smem,
                       cudaStream_t s, Follow follow) {
    cudaError_t e;
#define SHT_CALL(LV)                                                             \
    e = strided ? fft_launch(fx_forward_kernel<LV, true>, A, grid, smem, s, follow)          \
                : fft_launch(fx_forward_kernel<LV, false>, A, grid, smem, s, follow)
    SHT_FX_BODY(A.L, SHT_CALL)
#undef SHT_CALL
    return e;
}

cudaError_t fx_inverse(const InvArgs<double>& A, dim3 grid, size_t smem, cudaStream_t s, Follow follow) {
    if (A.mfactor1 != 1.0 && A.mfactor1 != 0.5) return cudaErrorInvalidValue;
    cudaError_t e;
#define SHT_CALL(LV) e = fft_launch(fx_inverse_kernel<LV>, A, grid, smem, s, follow)
    SHT_FX_BODY(A.L, SHT_CALL)
#undef SHT_CALL
    return e;
}

cudaError_t fx_forward_ragged(const RaggedFwd<double>& R, dim3 grid, size_t smem, cudaStream_t s, Follow follow) {
    return fft_launch(fx_forward_ragged_kernel, R, grid, smem, s, follow);
}

cudaError_t fx_inverse_ragged(const RaggedInv<double>& R, dim3 grid, size_t smem, cudaStream_t s, Follow follow) {
    if (R.a.mfactor1 != 1.0 && R.a.mfactor1 != 0.5) return cudaErrorInvalidValue;
    return fft_launch(fx_inverse_ragged_kernel, R, grid, smem, s, follow);
}

cudaError_t fx_forward_group(const FwdGroup<double>& G, int ctas, size_t smem, cudaStream_t s,
                             Follow follow) {
    return fft_launch(fx_forward_group_kernel, G, dim3(ctas), smem, s, follow);
}

cudaError_t fx_inverse_group(const InvGroup<double>& G, int ctas, size_t smem, cudaStream_t s,
                             Follow follow) {
    return fft_launch(fx_inverse_group_kernel, G, dim3(ctas), smem, s, follow);
}

}  // namespace sht
