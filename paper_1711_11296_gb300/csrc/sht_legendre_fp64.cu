// FP64 per-m Legendre contractions on the equatorially folded data
// (Eq. cc-quad and Eq. iLT in the parity form of Appendix B).
//
// Forward, per zonal wavenumber m and parity q (n - m = q mod 2):
//   X_n^m[c] = sum_{j < Jh} P~_n^m(mu_j) B_q[j][c]
// where B_0 = (X^m_S) w_j / I and B_1 = (X^m_A) w_j / I were written by the
// forward FFT (weights already folded in) and c runs over the 2F real
// columns (re, im of each field).
// Inverse, per m and q:
//   C_q[j][c] = sum_{n - m = q mod 2} P~_n^m(mu_j) X_n^m[c],
// the symmetric (q = 0) and antisymmetric (q = 1) halves that the inverse
// FFT unfolds into both hemispheres.
//
// These kernels run on the FP64 pipe: small transforms (legendre_small) with a
// thread per output, and those whose plan has no tensor-core tables
// (sht_slice64.cu) in tiles: a CTA computes a 32 x 64 output tile with 256
// threads (4 x 2 outputs each) over K chunks of 16 staged in shared memory,
// from a tile list {m, q, row0, col0} built once per plan.  The FP64 pipe,
// not memory, bounds both.
#include "sht_internal.h"

namespace sht {
namespace {

constexpr int BM = 32, BN = 64, BK = 16, NT = 256;

__device__ __forceinline__ int parity_rows(int N, int m, int q) {
    const int d = N - m - q;
    return d >= 0 ? d / 2 + 1 : 0;
}

__device__ __forceinline__ size_t dcoef_offset(int N, int m) {
    return (size_t)m * (N + 1) - (size_t)m * (m - 1) / 2;
}

// jmin (may be null): reduced transform (Sec. 4.1), per (m, parity) the
// first node with some |P~| >= 1e-16; the forward K loop starts at its
// K chunk, and inverse row tiles wholly before it are written as zero.
__device__ __forceinline__ void legendre_fwd_body(
    const double* __restrict__ pnm, int ldp, const double* __restrict__ work,
    double* __restrict__ spec, int4 t, int N, int Jh, int C, const int* __restrict__ jmin) {
    __shared__ double Ps[BK][BM + 1];
    __shared__ double Bs[BK][BN];
    const int m = t.x, q = t.y & 1, r0 = t.z, c0 = t.w;
    const int R = parity_rows(N, m, q);
    const size_t row0 = dcoef_offset(N, m) + q;     // packed row of n = m + q
    const double* B = work + ((size_t)(2 * m + q) * Jh) * C;
    const int tid = threadIdx.x, ty = tid >> 5, tx = tid & 31;
    double acc[4][2] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
    const int kstart = jmin ? (jmin[2 * m + q] / BK) * BK : 0;
    for (int k0 = kstart; k0 < Jh; k0 += BK) {
#pragma unroll
        for (int u = 0; u < (BM * BK) / NT; ++u) {
            const int e = tid + u * NT;
            const int rr = e / BK, kk = e % BK;
            const int r = r0 + rr, k = k0 + kk;
            Ps[kk][rr] = (r < R && k < Jh) ? pnm[(row0 + 2 * (size_t)r) * ldp + k] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < (BK * BN) / NT; ++u) {
            const int e = tid + u * NT;
            const int kk = e / BN, cc = e % BN;
            const int k = k0 + kk, c = c0 + cc;
            Bs[kk][cc] = (k < Jh && c < C) ? B[(size_t)k * C + c] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double a[4], b[2];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = Ps[kk][ty * 4 + i];
            b[0] = Bs[kk][tx];
            b[1] = Bs[kk][tx + 32];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[i][0] = fma(a[i], b[0], acc[i][0]);
                acc[i][1] = fma(a[i], b[1], acc[i][1]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = r0 + ty * 4 + i;
        if (r >= R) continue;
        double* out = spec + (row0 + 2 * (size_t)r) * C;
        if (c0 + tx < C) out[c0 + tx] = acc[i][0];
        if (c0 + tx + 32 < C) out[c0 + tx + 32] = acc[i][1];
    }
}

__device__ __forceinline__ void legendre_inv_body(
    const double* __restrict__ pnm, int ldp, const double* __restrict__ spec,
    double* __restrict__ work, int4 t, int N, int Jh, int C, const int* __restrict__ jmin) {
    __shared__ double Ps[BK][BM];
    __shared__ double Bs[BK][BN];
    const int m = t.x, q = t.y & 1, j0 = t.z, c0 = t.w;
    const int R = parity_rows(N, m, q);
    const size_t row0 = dcoef_offset(N, m) + q;
    const int tid = threadIdx.x, ty = tid >> 5, tx = tid & 31;
    double acc[4][2] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
    // (block-uniform: the loop holds barriers)
    const int kend = (jmin && j0 + BM <= jmin[2 * m + q]) ? 0 : R;
    for (int k0 = 0; k0 < kend; k0 += BK) {
#pragma unroll
        for (int u = 0; u < (BM * BK) / NT; ++u) {
            const int e = tid + u * NT;
            const int kk = e / BM, jj = e % BM;
            const int r = k0 + kk, j = j0 + jj;
            Ps[kk][jj] = (r < R && j < Jh) ? pnm[(row0 + 2 * (size_t)r) * ldp + j] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < (BK * BN) / NT; ++u) {
            const int e = tid + u * NT;
            const int kk = e / BN, cc = e % BN;
            const int r = k0 + kk, c = c0 + cc;
            Bs[kk][cc] = (r < R && c < C) ? spec[(row0 + 2 * (size_t)r) * C + c] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            double a[4], b[2];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = Ps[kk][ty * 4 + i];
            b[0] = Bs[kk][tx];
            b[1] = Bs[kk][tx + 32];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                acc[i][0] = fma(a[i], b[0], acc[i][0]);
                acc[i][1] = fma(a[i], b[1], acc[i][1]);
            }
        }
        __syncthreads();
    }
    double* W = work + ((size_t)(2 * m + q) * Jh) * C;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int j = j0 + ty * 4 + i;
        if (j >= Jh) continue;
        if (c0 + tx < C) W[(size_t)j * C + c0 + tx] = acc[i][0];
        if (c0 + tx + 32 < C) W[(size_t)j * C + c0 + tx + 32] = acc[i][1];
    }
}

__global__ void __launch_bounds__(NT) legendre_fwd_fp64_kernel(
    const double* __restrict__ pnm, int ldp, const double* __restrict__ work,
    double* __restrict__ spec, const int4* __restrict__ tiles, int N, int Jh, int C,
    const int* __restrict__ jmin) {
    legendre_fwd_body(pnm, ldp, work, spec, tiles[blockIdx.x], N, Jh, C, jmin);
}

__global__ void __launch_bounds__(NT) legendre_inv_fp64_kernel(
    const double* __restrict__ pnm, int ldp, const double* __restrict__ spec,
    double* __restrict__ work, const int4* __restrict__ tiles, int N, int Jh, int C,
    const int* __restrict__ jmin) {
    legendre_inv_body(pnm, ldp, spec, work, tiles[blockIdx.x], N, Jh, C, jmin);
}

// Small transforms (legendre_small): a thread per output, the same sums in the
// same order.  A tile's CTA computes 2048 products per K step whatever
// columns and rows there are (T31 x 1: 2 columns, at most 16 rows), and the
// slices take two launches and whole 16-column MMAs; here a K step is one
// product per output, bound by the FP64 pipe and, below it, by latency.
__global__ void __launch_bounds__(128) legendre_small_fp64_kernel(
    const double* __restrict__ pnm, int ldp, const double* in, double* __restrict__ out, int N,
    int Jh, int C, const int* __restrict__ jmin, int inverse, int wait) {
    grid_trigger();
    if (wait) grid_wait();
    const int m = blockIdx.x >> 1, q = blockIdx.x & 1;
    const int R = parity_rows(N, m, q);
    const size_t row0 = dcoef_offset(N, m) + q;
    const int o = blockIdx.y * 128 + threadIdx.x;
    const int row = o / C, c = o - row * C;
    if (row >= (inverse ? Jh : R)) return;
    const double* P = pnm + row0 * ldp;
    const size_t wrow = (size_t)(2 * m + q) * Jh;
    double acc = 0.0;
    if (!inverse) {
        const double* B = in + wrow * C + c;
        const double* A = P + 2 * (size_t)row * ldp;
#pragma unroll 8
        for (int k = jmin ? (jmin[2 * m + q] / BK) * BK : 0; k < Jh; ++k)
            acc = fma(__ldg(A + k), ld_dep(B + (size_t)k * C), acc);
        out[(row0 + 2 * (size_t)row) * C + c] = acc;
    } else {
        const double* B = in + row0 * C + c;
        const int kend = (jmin && row / BM * BM + BM <= jmin[2 * m + q]) ? 0 : R;
#pragma unroll 8
        for (int k = 0; k < kend; ++k)
            acc = fma(__ldg(P + 2 * (size_t)k * ldp + row), ld_dep(B + 2 * (size_t)k * C), acc);
        out[(wrow + row) * C + c] = acc;
    }
}

cudaError_t launch_small(const sht_plan_s* p, bool inverse, const double* in, double* out,
                         cudaStream_t s) {
    const int C = 2 * p->F, rows = inverse ? p->Jh : p->N / 2 + 1;
    const dim3 grid(2 * (p->N + 1), (rows * C + 127) / 128);
    const bool wait = short_launch((long long)grid.x * grid.y);
    return launch_kernel(legendre_small_fp64_kernel, grid, dim3(128), 0, s, wait, p->d_pnm, p->ldp,
                         in, out, p->N, p->Jh, C, p->d_jmin, inverse ? 1 : 0, wait ? 1 : 0);
}

}  // namespace

// us of the forward + inverse contraction, slices -> a thread per output: T31 x
// 10 30 -> 23, T63 x 20 40 -> 39, T95 x 8 51 -> 50, T127 x 2 55 -> 43; from
// 1.5e7 flops on T127 x 4 56 -> 57, T95 x 16 55 -> 72, T159 x 4 96 -> 100, T63
// x 64 47 -> 78, T200 x 4 116 -> 143, except for one field, whose 2 columns
// fill an eighth of an MMA: T319 x 1 274 -> 178, T639 x 1 1260 -> 1137.  (The
// tiles: T31 x 1 45, here 18.)
bool legendre_small(const sht_plan_s* p) {
    return p->F == 1 || 4.0 * (double)p->ncoef * p->Jh * p->F <= 1.5e7;
}

// Tile lists (host): forward tiles cover the parity rows of each (m, q);
// inverse tiles cover the Jh northern rows of each (m, q), including the
// empty parity (m = N, q = 1), whose output must still be written as zero.
void build_legendre_tiles(int N, int Jh, int C, std::vector<int4>& fwd,
                          std::vector<int4>& inv) {
    fwd.clear();
    inv.clear();
    for (int m = 0; m <= N; ++m) {
        for (int q = 0; q < 2; ++q) {
            const int d = N - m - q;
            const int R = d >= 0 ? d / 2 + 1 : 0;
            for (int r0 = 0; r0 < R; r0 += BM)
                for (int c0 = 0; c0 < C; c0 += BN) fwd.push_back(make_int4(m, q, r0, c0));
            for (int j0 = 0; j0 < Jh; j0 += BM)
                for (int c0 = 0; c0 < C; c0 += BN) inv.push_back(make_int4(m, q, j0, c0));
        }
    }
}

cudaError_t launch_legendre_fwd_fp64(const sht_plan_s* p, const double* work,
                                     double* spec, cudaStream_t s) {
    if (p->slice) return launch_legendre_slice64(p, false, work, spec, s);
    if (legendre_small(p)) return launch_small(p, false, work, spec, s);
    if (p->ntiles_fwd == 0) return cudaSuccess;
    legendre_fwd_fp64_kernel<<<p->ntiles_fwd, NT, 0, s>>>(
        p->d_pnm, p->ldp, work, spec, p->d_tiles_fwd, p->N, p->Jh, 2 * p->F, p->d_jmin);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_legendre_inv_fp64(const sht_plan_s* p, const double* spec,
                                     double* work, cudaStream_t s) {
    if (p->slice) return launch_legendre_slice64(p, true, spec, work, s);
    if (legendre_small(p)) return launch_small(p, true, spec, work, s);
    if (p->ntiles_inv == 0) return cudaSuccess;
    legendre_inv_fp64_kernel<<<p->ntiles_inv, NT, 0, s>>>(
        p->d_pnm, p->ldp, spec, work, p->d_tiles_inv, p->N, p->Jh, 2 * p->F, p->d_jmin);
    note_launch();
    return cudaGetLastError();
}

}  // namespace sht

namespace sht {
namespace {

// One thread per zonal wavenumber m: its tiles start after those of all
// m' < m (same order and geometry as build_legendre_tiles).
__global__ void fwd_tiles_kernel(int N, int C, int4* tiles) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m > N) return;
    const int nct = (C + BN - 1) / BN;
    auto rows = [&](int mm, int q) {
        const int d = N - mm - q;
        return d >= 0 ? d / 2 + 1 : 0;
    };
    long long off = 0;
    for (int mm = 0; mm < m; ++mm)
        off += (long long)((rows(mm, 0) + BM - 1) / BM + (rows(mm, 1) + BM - 1) / BM) * nct;
    for (int q = 0; q < 2; ++q) {
        const int R = rows(m, q);
        for (int r0 = 0; r0 < R; r0 += BM)
            for (int c0 = 0; c0 < C; c0 += BN) tiles[off++] = make_int4(m, q, r0, c0);
    }
}

}  // namespace

// Number of forward Legendre tiles for truncation N and C real columns.
int legendre_fwd_tile_count(int N, int C) {
    long long n = 0;
    const int nct = (C + BN - 1) / BN;
    for (int m = 0; m <= N; ++m)
        for (int q = 0; q < 2; ++q) {
            const int d = N - m - q;
            const int R = d >= 0 ? d / 2 + 1 : 0;
            n += (long long)((R + BM - 1) / BM) * nct;
        }
    return (int)n;
}

// Build the forward tile list on the device (no host memory involved).
cudaError_t launch_build_fwd_tiles(int N, int C, int4* tiles, cudaStream_t s) {
    const int threads = 128;
    fwd_tiles_kernel<<<(N + 1 + threads - 1) / threads, threads, 0, s>>>(N, C, tiles);
    return cudaGetLastError();
}

}  // namespace sht
