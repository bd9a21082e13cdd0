// FP64 Legendre contractions on the 5th-generation tensor cores, by an
// error-free split of both operands into 8-bit slices (Ozaki's scheme for
// matrix products, with balanced base-256 digits).
//
// The FP64 pipe of GB300 does 2 multiply-adds per clock and SM, so the
// 2.7e11 flops of a T639 x 256 pair take 241 ms on it at its full rate
// (sht_legendre_fp64.cu).  The tensor cores do about 1700 times as many
// BF16 products, and BF16 holds every integer up to 256 exactly.  Measured
// (us, forward / inverse contraction, FP64 pipe -> slices): T639 x 256
// 120600 / 117800 -> 6070 / 4720; T319 x 100 8530 / 8090 -> 558 / 445;
// T159 x 256 2721 / 2411 -> 254 / 225.
//
// Every row r of A (the P~ table) and every column c of B (the Fourier data
// or the spectrum) is scaled by a power of two to an integer of at most 2^sh (sh =
// 55; 54 and 53 for sums of more than 1000 and 4000 products), written with seven
// digits d_0 .. d_6 in [-128, 128], value = sum_a d_a 256^(6 - a).  An entry 2^-k
// of its row's or column's largest so keeps sh - k bits, an error of at most 2^-56
// of the largest at sh = 55; those within 2^-2 of it keep all 53.  Digit a is
// stored as the BF16 number d_a 2^(-8a) in slice a.  The products of equal a + b
// share an FP32 accumulator:
//   a + b = 0, 1, 2, 3, 4 | 5, 6, 7 together,
// 34 products of the 49 (the 15 left out are below 2^-60 of row times
// column maximum, under the rounding of the operands).
//
// The first five accumulators sum integers, exactly as long as these stay
// within 2^24.  Digits of ordinary data average out far below that, but those of
// a constant column and of the constant P~_0^0 do not (over the 776 nodes of
// T774 they reached 1.3 2^24, and the result was rounded at 6.6e-10).  So a
// tile's K slabs come in segments.  Accumulator a + b = s grows by at most
//   128 sum_k (|d_0| + .. + |d_s|) <= 128 sum_k (|d_0| + .. + |d_4|)
// of A's digits, whatever B holds, and table_segment_kernel ends a segment, when
// the plan is made, before any row's bound would pass 2^24 less what a carry
// leaves: after 12 slabs of 16 at the least, usually after about 25.  Between
// two segments the epilogue's warps carry: what accumulators 1 .. 4 hold beyond
// their own digit is added to the one before.  The first then holds the whole
// sum to within 2^9, at most K 2^(2 sh - 96), which sh keeps below 2^24.  The
// segments cost T639 x 256 5850 -> 6070 us forward (two a tile) and 4600 ->
// 4720 inverse, T319 x 100 547 -> 558 and 440 -> 445, T159 x 256 250 -> 254 and
// 222 -> 225 (one: the registers alone).
//
// The last accumulator rounds at 2^-24 of its leading term, 2^-62 of the maxima.
// The epilogue adds the six sums as a 64-bit integer, converts it once and
// scales it back, so an output carries the operands' rounding (2^-56 of the
// row and column maxima) and one final rounding: less than the sum of K
// FP64 products accumulates (T319 synthesis against 113-bit sums over the
// same table: 3.6e-16, FP64 pipe 6.6e-16).
//
// Per transform: slice_b_kernel reads the K x C operand of each (m, parity)
// problem once, finds the column exponents and writes the slices in the
// K-major core-matrix layout; slice_gemm_kernel multiplies, both operands
// arriving by bulk copies.  The slices of A are made once per plan.
#include <limits.h>
#include <stdlib.h>

#include <algorithm>
#include <new>
#include <vector>

#include "sht_internal.h"
#include "sht_tc.h"

namespace sht {

constexpr int kSlices = 7;
constexpr int kMaxJh = 4096;        // longest K
// segments of a problem, each of (2^24 - 2^16 - 2^7) / (5 128^2) = 203 or more K
// rows: 12 slabs
constexpr int kMaxSeg = kMaxJh / 16 / 12 + 1;

struct S64Prob {
    long long a_off;     // byte offset of the problem's A slices in the table
    long long b_off;     // byte offset of its B slices in the slice buffer
    long long src_off;   // double offset of B row 0 in the operand
    long long o_off;     // double offset of output row 0
    int R, R16;          // rows of A, rounded up to 16
    int K, nkt;          // depth, and its K slabs of 16
    int src_stride, o_stride;
    int ea_off;          // first row in the exponent table
    int sh;              // operands are integers of at most 2^sh
    int end0;            // end of the first segment (table_segment_kernel)
    int wide;            // the sum of the accumulators may need more than 63 bits
};

// One pass of slice_b + GEMM: problems [p0, p1), tiles [t0, t1).
struct S64Chunk { int p0, p1, t0, t1; };

struct S64Dir {
    bool mcols = true;              // the MMA's 128-wide M side holds columns (else rows)
    int tn = 80;                    // N width of the tiles
    unsigned char* table = nullptr; // A slices: per problem [K slab][slice][R16][16]
    int* ea = nullptr;              // exponent of every row of A
    int* seg = nullptr;             // [problem][kMaxSeg]: last K slab + 1 of its segments
    S64Prob* d_probs = nullptr;
    int4* d_tiles = nullptr;        // {problem, m0, n0, -}
    std::vector<S64Chunk> chunks;
    int maxK = 0;
};

struct Slice64 {
    S64Dir dir[2];                  // forward, inverse
    unsigned char* bbuf = nullptr;  // B slices of one chunk: [K slab][slice][C16][16]
    int* eb = nullptr;              // [problem][C16] column exponents
    int C16 = 0;
    size_t bytes = 0;               // device memory of all of it
};

namespace {

constexpr int TM = 128, TK = 16;            // MMA tile: M, K slab
constexpr int NACC = 6;                     // accumulators of TN TMEM columns
constexpr int TMEM_COLS = 512;
constexpr int M_SLICE = TM * TK * 2;        // bytes

// By the tile's N width: a stage holds the 14 slices of a K slab; as many
// stages as fit.
template <int TN> struct Cfg {
    static constexpr int N_SLICE = TN * TK * 2;
    static constexpr int STAGE = kSlices * (M_SLICE + N_SLICE);
    static constexpr int NSTAGE = (227 * 1024 - 256) / STAGE;
    static constexpr int NBAR = 2 * NSTAGE + 3;
    static constexpr int SMEM = NSTAGE * STAGE + 256;
    static_assert(8 * NBAR + 16 <= 256 && NACC * TN <= TMEM_COLS, "barriers and accumulators fit");
};

constexpr int NEPI = 512;                   // epilogue threads (16 warps)
constexpr int NT = NEPI + 64;               // + copy warp + MMA warp
constexpr int kNonFinite = INT_MAX;         // column exponent of Inf / NaN columns

// ---- slicing -------------------------------------------------------------

// |v| < 2^e for v with biased exponent field eb: e = max(eb, 1) - 1022.
__device__ __forceinline__ int exp_field(double v) {
    return (int)((__double_as_longlong(v) >> 52) & 0x7ff);
}

// v 2^(sh - e), e = exponent of the row or column maximum (biased field
// emax), rounded to nearest; |result| <= 2^sh.  Integer arithmetic: the FP64
// pipe would take longer than the memory traffic.
__device__ __forceinline__ long long to_fixed(double v, int emax, int sh) {
    const long long bits = __double_as_longlong(v);
    const int ex = (int)((bits >> 52) & 0x7ff);
    long long man = bits & 0xfffffffffffffll;
    if (ex) man |= 0x10000000000000ll;
    man <<= sh - 53;
    const int d = min(max(emax, 1) - max(ex, 1), 62);
    man = (man + ((1ll << d) >> 1)) >> d;
    return bits < 0 ? -man : man;
}

// The 16 bytes (one core-matrix row: 8 K values) of slice a of the
// integers x, biased by 128 in every digit so that digit a is
// (x >> 8 (6 - a)) & 0xff, minus 128 (the top digit has 9 bits).
__device__ __forceinline__ uint4 slice8(const long long (&x)[8], int a) {
    const float w = __uint_as_float((unsigned)(127 - 8 * a) << 23);   // 2^(-8a)
    unsigned h[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const unsigned dig = a == 0 ? (unsigned)(x[e] >> 48) & 0x1ffu
                                    : (unsigned)(x[e] >> (8 * (6 - a))) & 0xffu;
        // 2^23 + digit + 128, less 2^23 + 128; exact, as is the scaling, and
        // the 8 significant bits fill the upper half of the FP32 word
        h[e] = __float_as_uint((__uint_as_float(0x4B000000u | dig) - 8388736.f) * w);
    }
    return make_uint4(__byte_perm(h[0], h[1], 0x7632), __byte_perm(h[2], h[3], 0x7632),
                      __byte_perm(h[4], h[5], 0x7632), __byte_perm(h[6], h[7], 0x7632));
}

__device__ __forceinline__ long long bias(long long x) { return x + 0x80808080808080ll; }

// Byte offset of (row, K group k8 of the slab) within one slice.
__device__ __forceinline__ int core_off(int row, int k8) {
    return ((row >> 3) * 2 + k8) * 128 + (row & 7) * 16;
}

// Slices of the operand B of problems p0 + blockIdx.x, columns c0 + 32
// blockIdx.y + lane; warp w takes the groups of 8 K rows w, w + 16, ....
// NG > 0: at most NG groups per warp, held in registers between the
// exponent pass and the slicing; NG = 0: any K, read twice, the second time
// from the caches.  Latency and the 14 bytes written per value bound it, so
// the warps in flight count: one read with NG = 3 (92 registers, one CTA per
// SM) against two reads with three CTAs, contraction in us: T319 x 100 forward
// 564 / 546, inverse (NG = 2, 76 registers) 478 / 438, T639 x 256 inverse
// 4780 / 4593; where two CTAs fit, T159 x 256 forward (NG = 2) 249 / 268.
// Inverse: the Equator row (node Jh - 1), which the tiles leave out so that
// they cover J - 1 nodes in whole tiles, is summed here in FP64 (odd parity:
// P~(0) = 0).
template <int NG, bool INV>
__global__ void __launch_bounds__(512)
    slice_b_kernel(const double* B, const S64Prob* __restrict__ probs, int p0, int c0,
                   int C, int C16, unsigned char* __restrict__ out, int* __restrict__ eb,
                   const double* __restrict__ pnm, int ldp, int N, int Jh,
                   double* __restrict__ O, int wait) {
    __shared__ int red[16][32];
    __shared__ double redq[16][32];
    grid_trigger();
    if (wait) grid_wait();
    const int p = p0 + blockIdx.x;
    const S64Prob pr = probs[p];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int c = c0 + blockIdx.y * 32 + lane;
    const bool cin = c < C;
    const double* col = B + pr.src_off + c;
    auto load = [&](int k) -> double {
        return (k < pr.K && cin) ? ld_dep(col + (long long)k * pr.src_stride) : 0.0;
    };
    const int ng = 2 * pr.nkt;
    double v[NG > 0 ? 8 * NG : 8];
    int ex = 0;
    if constexpr (NG > 0) {
#pragma unroll
        for (int i = 0; i < NG; ++i)
#pragma unroll
            for (int e = 0; e < 8; ++e) v[8 * i + e] = load((w + 16 * i) * 8 + e);
#pragma unroll
        for (int i = 0; i < 8 * NG; ++i) ex = max(ex, exp_field(v[i]));
    } else {
        for (int g = w; g < ng; g += 16) {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = load(g * 8 + e);
#pragma unroll
            for (int e = 0; e < 8; ++e) ex = max(ex, exp_field(v[e]));
        }
    }
    if (INV) {
        double acc = 0.0;
        if ((p & 1) == 0) {
            const double* pe = pnm + coef_offset(N, p >> 1) * ldp + (Jh - 1);
            if constexpr (NG > 0) {
#pragma unroll
                for (int i = 0; i < NG; ++i)
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int k = (w + 16 * i) * 8 + e;
                        if (k < pr.K) acc = fma(__ldg(pe + 2 * (size_t)k * ldp), v[8 * i + e], acc);
                    }
            } else {
                for (int g = w; g < ng; g += 16)
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int k = g * 8 + e;
                        if (k < pr.K) acc = fma(__ldg(pe + 2 * (size_t)k * ldp), load(k), acc);
                    }
            }
        }
        redq[w][lane] = acc;
    }
    red[w][lane] = ex;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) ex = max(ex, red[i][lane]);
    if (w == 0 && c < C16)
        eb[(size_t)p * C16 + c] = ex == 0x7ff ? kNonFinite : max(ex, 1) - 1022;
    if (INV && w == 1 && cin) {
        double acc = redq[0][lane];
#pragma unroll
        for (int i = 1; i < 16; ++i) acc += redq[i][lane];
        O[pr.o_off + (long long)(Jh - 1) * pr.o_stride + c] = acc;
    }
    if (c >= C16) return;
    unsigned char* dst = out + pr.b_off;
    auto put = [&](int g, const double* x8) {
        long long x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = bias(to_fixed(x8[e], ex, pr.sh));
        unsigned char* d = dst + (long long)(g >> 1) * kSlices * C16 * 32 + core_off(c, g & 1);
#pragma unroll
        for (int a = 0; a < kSlices; ++a)
            *reinterpret_cast<uint4*>(d + (long long)a * C16 * 32) = slice8(x, a);
    };
    if constexpr (NG > 0) {
#pragma unroll
        for (int i = 0; i < NG; ++i)
            if (w + 16 * i < ng) put(w + 16 * i, v + 8 * i);
    } else {
        for (int g = w; g < ng; g += 16) {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = load(g * 8 + e);
            put(g, v);
        }
    }
}

// Row exponents (biased fields) of the table A of every problem.  Forward:
// rows n, K = nodes (a warp per row); inverse: rows = nodes, K = degrees (a
// thread per row).
__global__ void table_exp_kernel(const double* __restrict__ pnm, int ldp, int N,
                                 const S64Prob* __restrict__ probs, int inverse, int* ea) {
    const int p = blockIdx.x;
    const S64Prob pr = probs[p];
    const double* P = pnm + (coef_offset(N, p >> 1) + (p & 1)) * ldp;
    if (!inverse) {
        const int lane = threadIdx.x & 31;
        for (int r = threadIdx.x >> 5; r < pr.R16; r += blockDim.x >> 5) {
            int ex = 0;
            if (r < pr.R)
                for (int k = lane; k < pr.K; k += 32) ex = max(ex, exp_field(P[2 * (size_t)r * ldp + k]));
            ex = __reduce_max_sync(0xffffffffu, ex);
            if (lane == 0) ea[pr.ea_off + r] = ex;
        }
    } else {
        for (int r = threadIdx.x; r < pr.R16; r += blockDim.x) {
            int ex = 0;
            if (r < pr.R)
                for (int k = 0; k < pr.K; ++k) ex = max(ex, exp_field(P[2 * (size_t)k * ldp + r]));
            ea[pr.ea_off + r] = ex;
        }
    }
}

// Slices of A, one thread per (row, group of 8 K values).
__global__ void table_slice_kernel(const double* __restrict__ pnm, int ldp, int N,
                                   const S64Prob* __restrict__ probs, int inverse,
                                   const int* __restrict__ ea, unsigned char* __restrict__ out) {
    const int p = blockIdx.x;
    const S64Prob pr = probs[p];
    const double* P = pnm + (coef_offset(N, p >> 1) + (p & 1)) * ldp;
    const int ng = 2 * pr.nkt;
    const long long units = (long long)ng * pr.R16;
    for (long long u = (long long)blockIdx.y * blockDim.x + threadIdx.x; u < units;
         u += (long long)gridDim.y * blockDim.x) {
        // neighbouring threads: neighbouring rows, whose slices are adjacent (16
        // bytes each; forward, 64-byte pieces of the table's rows are read: with
        // neighbouring K groups instead 2.6 ms at T639, now 0.64)
        const int r = (int)(u % pr.R16), g = (int)(u / pr.R16);
        const int ex = ea[pr.ea_off + r];
        long long x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int k = g * 8 + e;
            const double v = (r < pr.R && k < pr.K)
                                 ? (inverse ? P[2 * (size_t)k * ldp + r] : P[2 * (size_t)r * ldp + k])
                                 : 0.0;
            x[e] = bias(to_fixed(v, ex, pr.sh));
        }
        unsigned char* d =
            out + pr.a_off + (long long)(g >> 1) * kSlices * pr.R16 * 32 + core_off(r, g & 1);
#pragma unroll
        for (int a = 0; a < kSlices; ++a)
            *reinterpret_cast<uint4*>(d + (long long)a * pr.R16 * 32) = slice8(x, a);
    }
}

// Ends of the K segments of every problem (see the top): the longest that keep
// 128 sum_k (|d_0| + .. + |d_4|) within 2^24 for every row, less the 2^16 + 2^7
// that a carry may leave in an accumulator.  One CTA per problem,
// a warp per row (forward) or a thread per row (inverse), as in
// table_exp_kernel.
__global__ void table_segment_kernel(const double* __restrict__ pnm, int ldp, int N,
                                     S64Prob* probs, int inverse, const int* __restrict__ ea,
                                     int* __restrict__ seg) {
    constexpr int LIM = ((1 << 24) - (1 << 16) - 128) / 128;
    __shared__ int end;
    const int p = blockIdx.x;
    const S64Prob pr = probs[p];
    const double* P = pnm + (coef_offset(N, p >> 1) + (p & 1)) * ldp;
    auto digits = [&](int r, int k) -> int {
        if (k >= pr.K) return 0;
        const double v = inverse ? P[2 * (size_t)k * ldp + r] : P[2 * (size_t)r * ldp + k];
        const long long x = bias(to_fixed(v, ea[pr.ea_off + r], pr.sh));
        int sum = abs((int)((x >> 48) & 0x1ff) - 128);
#pragma unroll
        for (int a = 1; a < 5; ++a) sum += abs((int)((x >> (8 * (6 - a))) & 0xff) - 128);
        return sum;
    };
    int n = 0;
    for (int q0 = 0; q0 < pr.nkt; ++n) {
        if (threadIdx.x == 0) end = pr.nkt;
        __syncthreads();
        if (pr.nkt - q0 <= 12) {
            // at most 5 128 a product: within the limit whatever the digits
            static_assert(12 * TK * 5 * 128 <= LIM, "twelve slabs need no look");
        } else if (!inverse) {
            const int lane = threadIdx.x & 31;
            for (int r = threadIdx.x >> 5; r < pr.R; r += blockDim.x >> 5) {
                int sum = 0;
                // two slabs at a time, eight loaded together
                for (int q = q0; q < pr.nkt && sum <= LIM; q += 8) {
                    int w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[i] = digits(r, (q + 2 * i) * TK + lane);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const bool in = sum <= LIM;
                        sum += __reduce_add_sync(0xffffffffu, w[i]);
                        if (in && sum > LIM && lane == 0) atomicMin(&end, q + 2 * i);
                    }
                }
            }
        } else {
            for (int r = threadIdx.x; r < pr.R; r += blockDim.x) {
                int sum = 0;
                for (int q = q0; q < pr.nkt; ++q) {
                    for (int e = 0; e < TK; ++e) sum += digits(r, q * TK + e);
                    if (sum > LIM) {
                        atomicMin(&end, q);
                        break;
                    }
                }
            }
        }
        __syncthreads();
        q0 = end;
        if (threadIdx.x == 0) {
            seg[(size_t)p * kMaxSeg + n] = q0;
            if (n == 0) probs[p].end0 = q0;
        }
        __syncthreads();   // end is written again only after all have read it
    }
}

// ---- the product ------------------------------------------------------------

struct S64Args {
    const unsigned char* table;
    const unsigned char* bbuf;
    const S64Prob* probs;
    const int4* tiles;
    int ntiles;
    double* O;
    const int* ea;
    const int* eb;
    const int* seg;
    const int* jmin;   // reduced transform (Sec. 4.1): first significant node per problem
    int inverse;
    int C, C16;
    int pairs;         // O is 16-byte aligned
    int wait;          // a dependent launch: wait for the kernel before
    int* status;
};

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&r)[4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr),
                 "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]));
}

// (hi 2^64 + lo) 2^k (two's complement) as a double, rounded once, by integer
// operations: the hardware conversion of 64-bit integers and FP64 compares
// run on the narrow FP64 pipe, which bound the epilogue (inverse contraction,
// us: T159 x 256 311 -> 222, T319 x 100 587 -> 478, T639 x 256 5137 -> 4781).
__device__ __forceinline__ double to_double(long long hi, unsigned long long lo, int k) {
    using u64 = unsigned long long;
    const u64 sign = (u64)hi & (1ull << 63);
    if (sign) {
        lo = 0 - lo;
        hi = ~hi + (lo == 0);
    }
    // u: the leading 64 bits, its last bit sticky
    u64 u = lo;
    if (hi) {
        const int l = __clzll(hi);   // >= 1
        u = ((u64)hi << l) | (lo >> (64 - l)) | ((lo << l) != 0);
        k += 64 - l;
    } else {
        if (lo == 0) return 0.0;
        const int l = __clzll((long long)lo);
        u <<= l;
        k -= l;
    }
    const u64 m = u >> 11;   // 53 bits
    const int e = 1086 + k, rem = (int)u & 0x7ff;
    if (e > 0 && e < 0x7ff)
        return __longlong_as_double(
            (long long)(sign | (((u64)(e - 1) << 52) + m + (rem + ((int)m & 1) > 0x400))));
    // below the normal range the scaling rounds (the last of the 53 bits is
    // sticky), above it gives infinity
    const double d = scalbn((double)(long long)(m | (rem != 0)), k + 11);
    return sign ? -d : d;
}

// Persistent CTAs, one per SM: 128 x TN tiles (M x N) with six FP32
// accumulators (480 of the 512 TMEM columns at TN = 80), K slabs of 16
// through a ring of 4 (TN = 80) to 6 (32) stages of 14 slices, 35 to 46 KB.
// Warps 0-15 the epilogue, warp 16 the bulk copies (a lane per slice), one
// thread of warp 17 the 34 MMAs of a stage.  The ring runs on across tiles, so
// the next tile's operands load during the epilogue.  An MMA reads 4 KB of M
// and TN 32 bytes of N from shared memory, 128 bytes per clock: 52 cycles at
// TN = 80 against 40 at the tensor rate, which bounds the main loop; the wider
// tile shares the M side among more columns (TN = 64 -> 80, us forward /
// inverse: T639 x 256 7114 / 8087 -> 6660 / 7522, T319 x 100 727 / 983 ->
// 687 / 845, T159 x 256 346 / 425 -> 316 / 362).  Where N never exceeds 64 or
// 32 the narrower configuration's deeper ring is faster (T200 x 20: TN = 80
// 100 / 119, 64 94 / 110).
// Six accumulators leave no room for a second set, so the MMAs wait while the
// epilogue reads them (or carries, between segments): it only forms the 64-bit
// sums in registers (60 a thread) before it hands them back, and converts,
// scales and stores beside the next tile's products.  With 16 warps against 8,
// and the sums by 32-bit multiply-adds: T639 x 256 6660 / 7500 -> 5780 / 5140,
// T319 x 100 685 / 845 -> 554 / 587, T159 x 256 316 / 362 -> 247 / 311 (8 warps
// alone 5820 / 5550, 562 / 676, 259 / 338).
template <bool MCOLS, int TN>
__global__ void __launch_bounds__(NT, 1) slice_gemm_kernel(const __grid_constant__ S64Args g) {
    using CF = Cfg<TN>;
    constexpr int NSTAGE = CF::NSTAGE, STAGE = CF::STAGE, NBAR = CF::NBAR, N_SLICE = CF::N_SLICE;
    grid_trigger();
    extern __shared__ __align__(1024) unsigned char s64_smem[];
    unsigned char* smem = s64_smem;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + NSTAGE * STAGE);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + NSTAGE * STAGE + 8 * NBAR);
    volatile int* abort_flag =
        reinterpret_cast<volatile int*>(smem + NSTAGE * STAGE + 8 * NBAR + 8);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar0 = smem_u32(bars);
    auto full = [&](int s) { return bar0 + 8u * s; };
    auto empty = [&](int s) { return bar0 + 8u * (NSTAGE + s); };
    const uint32_t done = bar0 + 8u * (2 * NSTAGE);   // a tile's accumulators complete
    const uint32_t acc_empty = done + 8u;             // read out by the epilogue
    const uint32_t fin = done + 16u;                  // every MMA of the CTA complete

    if (threadIdx.x == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), 1);
        }
        mbar_init(done, 1);
        mbar_init(acc_empty, NEPI);
        mbar_init(fin, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    if (g.wait) grid_wait();

    // first K slab and number of slabs of a tile (the reduced transform skips
    // forward slabs, and inverse tiles whose outputs are then zero, of nodes
    // before the first significant one)
    auto range = [&](const S64Prob& pr, const int4& t, int& kb) -> int {
        kb = 0;
        if (!g.jmin) return pr.nkt;
        const int j0 = g.jmin[t.x];
        if (g.inverse) {
            const int last = MCOLS ? t.z + TN : t.y + TM;
            return last <= j0 ? 0 : pr.nkt;
        }
        kb = min(j0 / TK, pr.nkt);
        return pr.nkt - kb;
    };
    auto aborted = [&]() { return __any_sync(0xffffffffu, *abort_flag != 0) != 0; };

    if (warp == NEPI / 32) {
        // ---- bulk copies: lane a < 7 slice a of M, lane 7 + a slice a of N ----
        uint32_t q = 0, issued = 0;
        bool ok = true;
        for (int tt = blockIdx.x; tt < g.ntiles && ok && !aborted(); tt += gridDim.x) {
            const int4 t = g.tiles[tt];
            const S64Prob pr = g.probs[t.x];
            int kb;
            const int nst = range(pr, t, kb);
            const int mrows = MCOLS ? g.C16 : pr.R16, nrows = MCOLS ? pr.R16 : g.C16;
            const int hm = min(TM, mrows - t.y), hn = min(TN, nrows - t.z);
            const unsigned char* mb =
                (MCOLS ? g.bbuf + pr.b_off : g.table + pr.a_off) + (long long)t.y * 32;
            const unsigned char* nb =
                (MCOLS ? g.table + pr.a_off : g.bbuf + pr.b_off) + (long long)t.z * 32;
            for (int li = 0; li < nst; ++li, ++q) {
                const int s = q % NSTAGE;
                if (lane == 0) {
                    ok = mbar_wait(empty(s), ((q / NSTAGE) & 1u) ^ 1u, abort_flag);
                    if (ok) mbar_expect_tx(full(s), (uint32_t)(kSlices * 32 * (hm + hn)));
                }
                ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
                if (!ok) break;
                issued = q + 1;
                const long long kt = kb + li;
                const uint32_t st = smem_u32(smem + s * STAGE);
                if (lane < kSlices) {
                    bulk_g2s(st + lane * M_SLICE, mb + (kt * kSlices + lane) * mrows * 32,
                             (uint32_t)hm * 32, full(s));
                } else if (lane < 2 * kSlices) {
                    const int a = lane - kSlices;
                    bulk_g2s(st + kSlices * M_SLICE + a * N_SLICE,
                             nb + (kt * kSlices + a) * nrows * 32, (uint32_t)hn * 32, full(s));
                }
                __syncwarp();
            }
        }
        // after an abort, let the copies in flight land (bounded)
        if (lane == 0 && *abort_flag) {
            for (uint32_t j = issued > (uint32_t)NSTAGE ? issued - NSTAGE : 0u; j < issued; ++j) {
                const long long t0 = clock64();
                while (!mbar_try(full(j % NSTAGE), (j / NSTAGE) & 1u) &&
                       clock64() - t0 < kWaitCycles) {
                }
            }
        }
    } else if (warp == NEPI / 32 + 1) {
        if (lane == 0) {
            uint32_t q = 0, nacc = 0;
            bool ok = true;
            for (int tt = blockIdx.x; tt < g.ntiles && ok && !*abort_flag; tt += gridDim.x) {
                const int4 t = g.tiles[tt];
                const S64Prob pr = g.probs[t.x];
                int kb;
                const int nst = range(pr, t, kb);
                if (nst == 0) continue;
                const int hn = min(TN, (MCOLS ? pr.R16 : g.C16) - t.z);
                const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                       ((uint32_t)(hn >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
                const int* seg = g.seg + (size_t)t.x * kMaxSeg;
                int end = pr.end0;
                while (end <= kb) end = *++seg;   // (the last ends at nkt > kb)
                bool first = true;                // of its segment
                for (int kt = kb; kt < pr.nkt; ++kt, ++q) {
                    if (first) {
                        if (nacc > 0 && !(ok = mbar_wait(acc_empty, (nacc - 1) & 1u, abort_flag)))
                            break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    }
                    const int s = q % NSTAGE;
                    if (!(ok = mbar_wait(full(s), (q / NSTAGE) & 1u, abort_flag))) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t st = smem_u32(smem + s * STAGE);
                    const uint64_t md = sdesc(st, 128, 256);
                    const uint64_t nd = sdesc(st + kSlices * M_SLICE, 128, 256);
#pragma unroll
                    for (int a = 0; a < kSlices; ++a) {
#pragma unroll
                        for (int b = 0; b < kSlices; ++b) {
                            if (a + b > 7) continue;
                            const int acc = a + b < NACC ? a + b : NACC - 1;
                            // (0, b) opens accumulator b
                            const uint32_t add = (kt > kb || !(a == 0 && b < NACC)) ? 1u : 0u;
                            mma_f16_rt(tmem + acc * TN, md + (uint64_t)(a * M_SLICE / 16),
                                       nd + (uint64_t)(b * N_SLICE / 16), idesc, add);
                        }
                    }
                    mma_commit(empty(s));
                    first = kt + 1 == end;
                    if (first) {
                        mma_commit(done);
                        ++nacc;
                        if (end < pr.nkt) end = *++seg;
                    }
                }
                if (!ok) break;
            }
            mma_commit(fin);
        }
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31 (the M
        // side), quarter w / 4 of the N columns ----
        uint32_t nacc = 0;
        bool ok = true;
        const int lq = warp & 3, quarter = warp >> 2;
        for (int tt = blockIdx.x; tt < g.ntiles && ok && !aborted(); tt += gridDim.x) {
            const int4 t = g.tiles[tt];
            const S64Prob pr = g.probs[t.x];
            int kb;
            const int nst = range(pr, t, kb);
            const bool have = nst > 0;
            constexpr int NI = TN / 16;   // groups of 4 columns
            const int i0 = quarter * (TN / 4), nb = t.z + i0;
            const int nv = MCOLS ? pr.R : g.C;
            const uint32_t acc = tmem + ((uint32_t)(32 * lq) << 16) + (uint32_t)i0;
            // wait for the accumulators of a segment
            auto take = [&]() {
                ok = mbar_wait(done, nacc & 1u, abort_flag);
                ok = __all_sync(0xffffffffu, ok) != 0;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            };
            auto hand_back = [&]() {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mbar_arrive(acc_empty);
                ++nacc;
            };
            // at the end of each segment but the last, carry (see the top)
            const int* seg = g.seg + (size_t)t.x * kMaxSeg;
            int end = pr.end0;
            while (have && end <= kb) end = *++seg;
            for (; have && ok && end < pr.nkt; end = *++seg) {
                take();
                if (!ok) break;
#pragma unroll
                for (int u = 0; u < NI; ++u) {
                    if (nb + 4 * u >= nv) continue;   // uniform over the warp
                    uint32_t r[NACC - 1][4];
#pragma unroll
                    for (int s = 0; s < NACC - 1; ++s)
                        tmem_ld4(acc + (uint32_t)(s * TN + 4 * u), r[s]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
#pragma unroll
                        for (int s = 1; s < NACC - 1; ++s) {
                            // to the nearest multiple of the unit of s - 1
                            const float a = __uint_as_float(r[s][i]);
                            const float big = 12582912.f / (float)(1ull << (8 * (s - 1)));
                            const float c = (a + big) - big;
                            r[s - 1][i] = __float_as_uint(__uint_as_float(r[s - 1][i]) + c);
                            r[s][i] = __float_as_uint(a - c);
                        }
                    }
#pragma unroll
                    for (int s = 0; s < NACC - 1; ++s)
                        tmem_st4(acc + (uint32_t)(s * TN + 4 * u), r[s]);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                hand_back();
            }
            if (have && ok) take();
            const int im = t.y + 32 * lq + lane;           // this lane's M index
            const int mv = MCOLS ? g.C : pr.R;
            const bool mok = im < mv && ok;
            const int* ebp = g.eb + (size_t)t.x * g.C16;
            const int* eap = g.ea + pr.ea_off;
            auto row_exp = [&](int r) { return max(__ldg(eap + r), 1) - 1022; };
            const int em = mok ? (MCOLS ? ld_dep(ebp + im) : row_exp(im)) : 0;
            double* om = g.O + pr.o_off + (MCOLS ? (long long)im : (long long)im * pr.o_stride);
            const int k0 = 56 - 2 * pr.sh;
            // The accumulators become 64-bit integers in registers first and
            // go back to the MMAs; conversion, scaling and stores run beside
            // the next tile's products.
            long long T[NI][4];
            int lead[NI][4];
            if (have) {
#pragma unroll
                for (int u = 0; u < NI; ++u) {
                    if (nb + 4 * u >= nv || !ok) continue;   // uniform over the warp
                    uint32_t r[NACC][4];
#pragma unroll
                    for (int s = 0; s < NACC; ++s)
                        tmem_ld4(acc + (uint32_t)(s * TN + 4 * u), r[s]);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        // sum of the accumulators in units of 2^-40 (the first
                        // apart where 64 bits may not hold it)
                        int d[NACC];
#pragma unroll
                        for (int s = 0; s < NACC; ++s)
                            d[s] = __float2int_rn(__uint_as_float(r[s][i]) *
                                                  (float)(1ull << (8 * s)));
                        lead[u][i] = d[0];
                        using u64 = unsigned long long;
                        T[u][i] = (long long)(((u64)((pr.wide ? 0 : d[0]) * 256ll + d[1]) << 32) +
                                              ((u64)(d[2] * 256ll + d[3]) << 16) +
                                              (u64)(d[4] * 256ll + d[5]));
                    }
                }
                if (ok) hand_back();
            }
            auto value = [&](int u, int i, int in) -> double {
                if (!have) return 0.0;
                const int en = MCOLS ? row_exp(in) : ld_dep(ebp + in);
                if ((MCOLS ? em : en) == kNonFinite)
                    return __longlong_as_double(0x7ff8000000000000ll);
                using u64 = unsigned long long;
                long long hi = T[u][i] >> 63;
                u64 lo = (u64)T[u][i];
                if (pr.wide) {
                    const u64 add = (u64)(long long)lead[u][i] << 40;
                    hi += (long long)(lead[u][i] >> 24) + (lo + add < add);
                    lo += add;
                }
                return to_double(hi, lo, em + en + k0);
            };
#pragma unroll
            for (int u = 0; u < NI; ++u) {
                const int n0 = nb + 4 * u;
                if (!mok) continue;
                if constexpr (MCOLS) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (n0 + i < nv) om[(n0 + i) * (long long)pr.o_stride] = value(u, i, n0 + i);
                } else {
                    // columns come in pairs (re, im), adjacent in the lane's row
#pragma unroll
                    for (int i = 0; i < 4; i += 2) {
                        if (n0 + i >= nv) continue;
                        const double x = value(u, i, n0 + i), y = value(u, i + 1, n0 + i + 1);
                        if (g.pairs) {
                            *reinterpret_cast<double2*>(om + n0 + i) = make_double2(x, y);
                        } else {
                            om[n0 + i] = x;
                            om[n0 + i + 1] = y;
                        }
                    }
                }
            }
        }
    }
    if (*abort_flag && threadIdx.x == 0 && g.status) atomicOr(g.status, 1);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        const long long t0 = clock64();
        while (!mbar_try(fin, 0) && clock64() - t0 < kWaitCycles) {
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(TMEM_COLS)
                     : "memory");
    }
}

// ---- host ---------------------------------------------------------------------

constexpr size_t kChunkBytes = 1ull << 30;   // B slices of one pass

struct HostDir {
    std::vector<S64Prob> probs;
    std::vector<int4> tiles;
    long long table_bytes = 0, ea_rows = 0;
    size_t bbytes = 0;   // the largest chunk's B slices
};

void build_dir(int N, int Jh, int C, bool inverse, S64Dir& d, HostDir& h) {
    const int nprob = 2 * (N + 1), C16 = (C + 15) / 16 * 16;
    h.probs.assign(nprob, S64Prob{});
    long long mac_cols = 0, mac_rows = 0;   // padded MMA work of either orientation
    for (int p = 0; p < nprob; ++p) {
        const int m = p >> 1, q = p & 1, dd = N - m - q;
        const int Rn = dd >= 0 ? dd / 2 + 1 : 0;   // degrees of this parity
        const long long row0 = (long long)coef_offset(N, m) + q;
        S64Prob& s = h.probs[p];
        s.R = inverse ? Jh - 1 : Rn;
        s.K = inverse ? Rn : Jh;
        s.R16 = (s.R + 15) / 16 * 16;
        s.nkt = (s.K + TK - 1) / TK;
        // K products of the operands are at most K 2^(2 sh - 96) in the first
        // accumulator's units, within the 2^24 that FP32 adds exactly (the
        // others: table_segment_kernel); the sum of the six fits a 64-bit
        // integer (K 2^14 2^40 and the rest below 2^63) up to K = 480
        s.sh = s.K <= 1000 ? 55 : s.K <= 4000 ? 54 : 53;
        s.wide = s.K > 480;
        s.src_off = inverse ? row0 * C : (long long)p * Jh * C;
        s.src_stride = inverse ? 2 * C : C;
        s.o_off = inverse ? (long long)p * Jh * C : row0 * C;
        s.o_stride = inverse ? C : 2 * C;
        s.a_off = h.table_bytes;
        h.table_bytes += (long long)s.nkt * kSlices * s.R16 * 32;
        s.ea_off = (int)h.ea_rows;
        h.ea_rows += s.R16;
        d.maxK = std::max(d.maxK, s.K);
        mac_cols += (long long)s.nkt * ((C16 + TM - 1) / TM * TM) * s.R16;
        mac_rows += (long long)s.nkt * ((s.R16 + TM - 1) / TM * TM) * C16;
    }
    // columns on the M side also store whole rows, worth some padding (T319 x
    // 100 inverse, 2 % more work: 809 us with rows, 676 with columns; T200 x
    // 20 forward, 20 % more: 81 and 97)
    d.mcols = mac_cols * 10 <= mac_rows * 11;
    int nmax = C16;
    if (d.mcols) {
        nmax = 0;
        for (const S64Prob& s : h.probs) nmax = std::max(nmax, s.R16);
    }
    d.tn = nmax <= 32 ? 32 : nmax <= 64 ? 64 : 80;
    S64Chunk ch{0, 0, 0, 0};
    size_t used = 0;
    for (int p = 0; p < nprob; ++p) {
        S64Prob& s = h.probs[p];
        const size_t need = (size_t)s.nkt * kSlices * C16 * 32;
        if (used > 0 && used + need > kChunkBytes) {
            ch.p1 = p;
            ch.t1 = (int)h.tiles.size();
            d.chunks.push_back(ch);
            ch = S64Chunk{p, p, ch.t1, ch.t1};
            used = 0;
        }
        s.b_off = (long long)used;
        used += need;
        h.bbytes = std::max(h.bbytes, used);
        const int mr = d.mcols ? C16 : s.R16, nr = d.mcols ? s.R16 : C16;
        for (int m0 = 0; m0 < mr; m0 += TM)
            for (int n0 = 0; n0 < nr; n0 += d.tn) h.tiles.push_back(make_int4(p, m0, n0, 0));
    }
    ch.p1 = nprob;
    ch.t1 = (int)h.tiles.size();
    d.chunks.push_back(ch);
}

template <bool INV>
cudaError_t launch_slice_b(int maxK, cudaStream_t s, const double* B, const S64Prob* probs, int p0,
                           int np, int C, int C16, unsigned char* out, int* eb, const double* pnm,
                           int ldp, int N, int Jh, double* O) {
    using Fn = void (*)(const double*, const S64Prob*, int, int, int, int, unsigned char*, int*,
                        const double*, int, int, int, double*, int);
    // in registers where two CTAs still fit an SM
    const int ng = (maxK + 127) / 128;
    const Fn fn = ng == 1            ? slice_b_kernel<1, INV>
                  : ng == 2 && !INV ? slice_b_kernel<2, false>
                                    : slice_b_kernel<0, INV>;
    // (a grid's second dimension holds 65535 blocks, 2^20 fields)
    for (int y0 = 0, ny = (C16 + 31) / 32; y0 < ny; y0 += 65535) {
        const dim3 grid(np, std::min(ny - y0, 65535));
        const bool wait = short_launch((long long)grid.x * grid.y);
        const cudaError_t e =
            launch_kernel(fn, grid, dim3(512), 0, s, wait, B, probs, p0, 32 * y0, C, C16, out, eb,
                          pnm, ldp, N, Jh, O, wait ? 1 : 0);
        if (e) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_dir(const sht_plan_s* p, bool inverse, const double* B, double* O,
                       cudaStream_t s) {
    const Slice64* sl = p->slice;
    const S64Dir& d = sl->dir[inverse ? 1 : 0];
    const int C = 2 * p->F;
    using Gemm = void (*)(const S64Args);
    Gemm fn;
    int smem;
    if (d.tn == 32) {
        fn = d.mcols ? slice_gemm_kernel<true, 32> : slice_gemm_kernel<false, 32>;
        smem = Cfg<32>::SMEM;
    } else if (d.tn == 64) {
        fn = d.mcols ? slice_gemm_kernel<true, 64> : slice_gemm_kernel<false, 64>;
        smem = Cfg<64>::SMEM;
    } else {
        fn = d.mcols ? slice_gemm_kernel<true, 80> : slice_gemm_kernel<false, 80>;
        smem = Cfg<80>::SMEM;
    }
    cudaError_t e = ensure_smem((const void*)fn, smem);
    if (e) return e;
    for (const S64Chunk& c : d.chunks) {
        const int np = c.p1 - c.p0;
        if (inverse)
            e = launch_slice_b<true>(d.maxK, s, B, d.d_probs, c.p0, np, C, sl->C16, sl->bbuf,
                                     sl->eb, p->d_pnm, p->ldp, p->N, p->Jh, O);
        else
            e = launch_slice_b<false>(d.maxK, s, B, d.d_probs, c.p0, np, C, sl->C16, sl->bbuf,
                                      sl->eb, p->d_pnm, p->ldp, p->N, p->Jh, O);
        if (e) return e;
        S64Args g;
        g.table = d.table;
        g.bbuf = sl->bbuf;
        g.probs = d.d_probs;
        g.tiles = d.d_tiles + c.t0;
        g.ntiles = c.t1 - c.t0;
        g.O = O;
        g.ea = d.ea;
        g.eb = sl->eb;
        g.seg = d.seg;
        g.jmin = p->d_jmin;
        g.inverse = inverse ? 1 : 0;
        g.C = C;
        g.C16 = sl->C16;
        g.status = p->d_status;
        g.pairs = ((uintptr_t)O & 15) == 0;
        g.wait = short_launch(g.ntiles) ? 1 : 0;
        if (g.ntiles == 0) continue;
        const int ctas = std::min(g.ntiles, p->num_sms);
        e = launch_kernel(fn, dim3(ctas), dim3(NT), smem, s, g.wait != 0, g);
        if (e) return e;
    }
    return cudaSuccess;
}

}  // namespace

bool slice64_takes(const sht_plan_s* p) { return !legendre_small(p) && p->Jh <= kMaxJh; }

size_t slice64_bytes(const sht_plan_s* p) { return p->slice ? p->slice->bytes : 0; }

// The slice tables of an FP64 plan that slice64_takes.  share > 0: only if they
// take no more than 1 / share of the device's free memory.  Without them (also
// when an allocation fails, cudaErrorMemoryAllocation) the plan's contractions
// stay on the FP64 pipe.
cudaError_t slice64_create(sht_plan_s* p, int share, const DeviceAlloc& alloc, cudaStream_t s) {
    if (!slice64_takes(p) || p->slice) return cudaSuccess;
    Slice64* sl = new (std::nothrow) Slice64();
    if (!sl) return cudaErrorMemoryAllocation;
    p->slice = sl;
    const int C = 2 * p->F, nprob = 2 * (p->N + 1);
    sl->C16 = (C + 15) / 16 * 16;
    HostDir h[2];
    struct Part { void** ptr; size_t bytes; };
    std::vector<Part> parts;
    try {
        for (int i = 0; i < 2; ++i) build_dir(p->N, p->Jh, C, i == 1, sl->dir[i], h[i]);
        parts.reserve(12);
    } catch (const std::bad_alloc&) {
        slice64_destroy(p);
        return cudaErrorMemoryAllocation;
    }
    auto part = [&](auto& ptr, size_t bytes) {
        parts.push_back({reinterpret_cast<void**>(&ptr), bytes});
        sl->bytes += bytes;
    };
    part(sl->bbuf, std::max(h[0].bbytes, h[1].bbytes));
    part(sl->eb, (size_t)nprob * sl->C16 * sizeof(int));
    for (int i = 0; i < 2; ++i) {
        S64Dir& d = sl->dir[i];
        part(d.table, (size_t)h[i].table_bytes + 16);
        part(d.ea, (size_t)(h[i].ea_rows + 1) * sizeof(int));
        part(d.seg, (size_t)nprob * kMaxSeg * sizeof(int));
        part(d.d_probs, nprob * sizeof(S64Prob));
        part(d.d_tiles, (h[i].tiles.size() + 1) * sizeof(int4));
    }
    cudaError_t e = cudaSuccess;
    if (share > 0) {
        size_t avail = 0, total = 0;
        e = cudaMemGetInfo(&avail, &total);
        // (tests: SHT_INJECT_FREE_BYTES stands for what is free)
        if (const char* v = getenv("SHT_INJECT_FREE_BYTES")) avail = (size_t)strtoull(v, nullptr, 10);
        if (e == cudaSuccess && sl->bytes > avail / share) {
            slice64_destroy(p);
            return cudaSuccess;
        }
    }
    for (const Part& q : parts)
        if (e == cudaSuccess) e = alloc(q.ptr, q.bytes);
    if (e != cudaSuccess) {
        slice64_destroy(p);
        cudaGetLastError();
        return e;
    }
    for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
        S64Dir& d = sl->dir[i];
        e = cudaMemcpyAsync(d.d_probs, h[i].probs.data(), nprob * sizeof(S64Prob),
                            cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(d.d_tiles, h[i].tiles.data(), h[i].tiles.size() * sizeof(int4),
                                cudaMemcpyHostToDevice, s);
        if (e != cudaSuccess) break;
        table_exp_kernel<<<nprob, 256, 0, s>>>(p->d_pnm, p->ldp, p->N, d.d_probs, i, d.ea);
        table_slice_kernel<<<dim3(nprob, 8), 256, 0, s>>>(p->d_pnm, p->ldp, p->N, d.d_probs, i,
                                                         d.ea, d.table);
        table_segment_kernel<<<nprob, 256, 0, s>>>(p->d_pnm, p->ldp, p->N, d.d_probs, i, d.ea,
                                                   d.seg);
        e = cudaGetLastError();
    }
    // (the host lists above must outlive the copies)
    const cudaError_t es = cudaStreamSynchronize(s);
    return e == cudaSuccess ? es : e;
}

void slice64_destroy(sht_plan_s* p) {
    Slice64* sl = p->slice;
    if (!sl) return;
    if (sl->bbuf) cudaFree(sl->bbuf);
    if (sl->eb) cudaFree(sl->eb);
    for (S64Dir& d : sl->dir) {
        void* ptrs[] = {d.table, d.ea, d.seg, d.d_probs, d.d_tiles};
        for (void* q : ptrs)
            if (q) cudaFree(q);
    }
    delete sl;
    p->slice = nullptr;
}

cudaError_t launch_legendre_slice64(const sht_plan_s* p, bool inverse, const double* in,
                                    double* out, cudaStream_t s) {
    return launch_dir(p, inverse, in, out, s);
}

}  // namespace sht
