// pca.cu -- the PCA start of Algorithm 1 (Sec. IV of Kvinge et al.,
// arXiv:1807.03425): the first basis is made of the top k left singular
// vectors of the n x p matrix S whose columns are the unit secants, i.e. the
// eigenvectors of C = S S^T with the k largest eigenvalues.
//
// S is never formed (p = N(N-1)/2 columns).  C is built in FP64 through the
// weighted graph Laplacian of the pairs:
//     C = sum_{i<j kept} (x_i - x_j)(x_i - x_j)^T / d_ij^2 = Xc^T R,
//     R_i = sum_{j kept} w_ij (x_i - x_j),  w_ij = 1/d_ij^2,  Xc = X - mean,
// (sum_i R_i = 0, so centring X is free and keeps the terms small).  Three
// kernels: FP64 inverse squared lengths from explicit differences (upper
// triangle, 64 x 64 tiles, 0 for excluded pairs: d = 0, Sec. II, or d < eps,
// Sec. VII); the rows R_i (every block owns one block of rows and walks all
// column blocks, reading the stored upper triangle transposed where needed,
// so no atomics and a fixed summation order); and C = Xc^T R.
//
// The n x n symmetric eigenproblem (the paper calls cuSolver's SVD for this
// step, Sec. V) is solved here by the cyclic Jacobi method in FP64 (Golub
// and Van Loan, Matrix Computations, Sec. 8.5): sweeps of plane rotations,
// each zeroing one off-diagonal entry (p, q) with the rotation of the 2 x 2
// symmetric Schur decomposition, in the round-robin ("tournament") order of
// the parallel variant: n' - 1 rounds of n'/2 disjoint pairs per sweep (n'
// = n rounded up to even; an odd n's extra index pairs with nobody), so
// one round is one independent rotation per pair, applied to A from both
// sides and to the accumulated vectors V.  Sweeps stop when the
// off-diagonal Frobenius norm is below 4 n 2^-53 of the whole (quadratic
// convergence: typically 6 to 10 sweeps), or after 40.
#include "sap_internal.cuh"
#include "colmean.cuh"
#include "../../include/sap.h"

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

namespace cg = cooperative_groups;

namespace sap {

// engine accessors (capi.cu)
cudaStream_t handle_stream(sap_handle h);
int64_t handle_n_points(sap_handle h);
int handle_n_dim(sap_handle h);
const float *handle_x32(sap_handle h);
const double *handle_x64(sap_handle h);
double handle_eps2(sap_handle h);
int handle_sms(sap_handle h);
const float *handle_nu(sap_handle h);  // ||x_i - mean||, rounded up (FP32/BF16 data)
sap_status handle_fail(sap_handle h, sap_status s, const char *msg);

namespace {

constexpr int PT = 64;   // points per block side
constexpr int PC = 32;   // coordinates per chunk

template <typename TX>
__device__ __forceinline__ double ldx(const TX *X, size_t i)
{
    return (double)X[i];
}

// Inverse squared lengths of the pairs of one upper-triangle tile (I <= J).
template <typename TX>
__global__ void __launch_bounds__(256) w64_kernel(const TX *X, int N, int n, const int2 *tiles, double eps2,
                                                  double *w)
{
    __shared__ double xi[PC][PT + 1], xj[PC][PT + 1];
    const int2 IJ = tiles[blockIdx.x];
    const int i0 = IJ.x * PT, j0 = IJ.y * PT;
    const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;  // 4 x 4 pairs each
    double d2[4][4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) d2[p][q] = 0.0;
    for (int c0 = 0; c0 < n; c0 += PC) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < PT * PC; idx += 256) {
            const int r = idx / PC, l = idx % PC;
            const bool inl = c0 + l < n;
            xi[l][r] = (i0 + r < N && inl) ? ldx(X, (size_t)(i0 + r) * n + c0 + l) : 0.0;
            xj[l][r] = (j0 + r < N && inl) ? ldx(X, (size_t)(j0 + r) * n + c0 + l) : 0.0;
        }
        __syncthreads();
        const int lc = min(PC, n - c0);
        for (int l = 0; l < lc; ++l)
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const double D = xi[l][tr * 4 + p] - xj[l][tc * 4 + q];
                    d2[p][q] = fma(D, D, d2[p][q]);
                }
    }
    double *out = w + (size_t)blockIdx.x * PT * PT;
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + tr * 4 + p, j = j0 + tc * 4 + q;
            const double d = d2[p][q];
            const bool kept = i < j && j < N && d != 0.0 && !(d < eps2);
            out[(tr * 4 + p) * PT + tc * 4 + q] = kept ? 1.0 / d : 0.0;
        }
}

__device__ __forceinline__ long long tile_of(int I, int J, int nb)
{
    return (long long)I * nb - (long long)I * (I - 1) / 2 + (J - I);
}

// R_i = sum_j w_ij (x_i - x_j) for the 64 rows of block I and the
// coordinates c0 .. c0 + 31 (blockIdx.y); thread: one row, 8 coordinates.
template <typename TX>
__global__ void __launch_bounds__(256) lap_rows_kernel(const TX *X, int N, int n, const double *w, int nb,
                                                       double *R)
{
    __shared__ double wt[PT][PT + 1];
    __shared__ double xs[PT][PC + 1];
    const int I = blockIdx.x, c0 = blockIdx.y * PC;
    const int r = threadIdx.x & (PT - 1), g = threadIdx.x >> 6;  // 4 groups of 8 coordinates
    const int i = I * PT + r;
    double xi[8], acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int l = c0 + g * 8 + q;
        xi[q] = (i < N && l < n) ? ldx(X, (size_t)i * n + l) : 0.0;
        acc[q] = 0.0;
    }
    for (int J = 0; J < nb; ++J) {
        __syncthreads();
        const double *tw = w + tile_of(min(I, J), max(I, J), nb) * (PT * PT);
        for (int idx = threadIdx.x; idx < PT * PT; idx += 256) {
            const int a = idx / PT, b = idx % PT;  // a: row of this block, b: row of block J
            double v;
            if (I < J) v = tw[a * PT + b];
            else if (I > J) v = tw[b * PT + a];
            else v = a < b ? tw[a * PT + b] : (a > b ? tw[b * PT + a] : 0.0);
            wt[a][b] = v;
        }
        for (int idx = threadIdx.x; idx < PT * PC; idx += 256) {
            const int b = idx / PC, l = idx % PC;
            const int j = J * PT + b;
            xs[b][l] = (j < N && c0 + l < n) ? ldx(X, (size_t)j * n + c0 + l) : 0.0;
        }
        __syncthreads();
        for (int b = 0; b < PT; ++b) {
            const double wv = wt[r][b];
            if (wv == 0.0) continue;
#pragma unroll
            for (int q = 0; q < 8; ++q) acc[q] = fma(wv, xi[q] - xs[b][g * 8 + q], acc[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int l = c0 + g * 8 + q;
        if (i < N && l < n) R[(size_t)i * n + l] = acc[q];
    }
}

// ---- FP32/BF16 data: the same two kernels in FP32 pairs (double-float)
//
// FP64 issues at 1/64 of the FP32 rate here, and the two kernels above are
// bound by it (12.6 ms and 39 ms at N = 8192, n = 100).  With FP32 points the
// difference of two coordinates is an exact FP32 pair s + e, so lengths and
// weighted differences can be formed with error-free FP32 steps (18
// operations instead of two FP64 ones: 2.2 ms and 7.2 ms), accurate to a few
// 2^-48 of the running sums.  That is enough where w = 1/d^2 is moderate; the
// Laplacian's rounding error is carried by the short secants, whose terms (of
// size 1/d) cancel between neighbours: a rounding of R_i reaches S S^T times
// x_i, so the pairs whose d is below a sixteenth of the larger of their own
// ||x - mean|| keep FP64 arithmetic throughout.  (A cut against the largest
// norm of all points let one point a hundred times farther out make every
// secant short: 87 ms instead of 13.)  Measured against the
// compensated sum of the secants' outer products, over ten families of curves
// and scenes (700 to 8192 points, n = 8 .. 160, 4 to 10 draws each), the
// vectors' errors are 0.4 to 1.1 times those of the FP64 form (geometric means
// of the largest entry; 8.1e-14 against 7.8e-14 at N = 8192, n = 100, where
// both come from the product with Xc), the values' 0.2 to 1.2 times.
// N = 8192, n = 100, whole start, FP64 form -> this: a smooth curve 62.2 ->
// 13.4 ms, with one point a hundred times farther out 62.3 -> 13.4, fifty
// tight clusters 65.3 -> 43.9, two tight clusters 62.2 -> 50.4.
//
// The FP64 operations of the short secants: the difference of two FP32
// numbers is an exact FP32 sum and remainder, widened by integer operations,
// so a term takes one FP64 addition and one multiply-add (one multiply-add
// where the difference is exact in FP32, as it is for close numbers), not
// more than the FP64 kernels above take.
//
// A pair's 8 bytes hold either the FP64 w (sign bit 0; 0.0: excluded) or,
// sign bit 1, the FP32 pair: -wh in the high word, wl in the low one.

__device__ __forceinline__ void two_diff(float a, float b, float &s, float &e)
{
    s = __fsub_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb));
}
__device__ __forceinline__ void add_pair(float &hi, float &lo, float p, float pe)
{
    const float s = __fadd_rn(hi, p);
    const float bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(e, pe));
}

// Shared-memory rows that are read 16 bytes at a time: the array and every
// row start on such a boundary.
template <int ROWS, int COLS>
struct __align__(16) Staged {
    float v[ROWS][COLS];
    static_assert(COLS * sizeof(float) % 16 == 0, "rows are read as float4");
};

// x - y in FP64 from the two_diff parts (an overflow of the FP32 difference
// takes the conversions).
__device__ __forceinline__ double diff64(float x, float y, float s, float e)
{
    if (!(fabsf(s) < INFINITY)) return (double)x - (double)y;
    return e == 0.f ? widen(s) : widen(s) + widen(e);
}

__global__ void __launch_bounds__(256) w_pair_kernel(const float *X, int N, int n, const int2 *tiles, double eps2,
                                                     const float *nu, unsigned long long *w)
{
    __shared__ Staged<PC, PT + 4> xi_, xj_;
    auto &xi = xi_.v, &xj = xj_.v;
    const int2 IJ = tiles[blockIdx.x];
    const int i0 = IJ.x * PT, j0 = IJ.y * PT;
    const int tr = threadIdx.x >> 4, tc = threadIdx.x & 15;  // 4 x 4 pairs each
    float hi[4][4], lo[4][4];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) hi[p][q] = lo[p][q] = 0.f;
    for (int c0 = 0; c0 < n; c0 += PC) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < PT * PC; idx += 256) {
            const int r = idx / PC, l = idx % PC;
            const bool inl = c0 + l < n;
            xi[l][r] = (i0 + r < N && inl) ? X[(size_t)(i0 + r) * n + c0 + l] : 0.f;
            xj[l][r] = (j0 + r < N && inl) ? X[(size_t)(j0 + r) * n + c0 + l] : 0.f;
        }
        __syncthreads();
        const int lc = min(PC, n - c0);
#pragma unroll 2
        for (int l = 0; l < lc; ++l) {
            const float4 a4 = *reinterpret_cast<const float4 *>(&xi[l][tr * 4]);
            const float4 b4 = *reinterpret_cast<const float4 *>(&xj[l][tc * 4]);
            const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float s, e;
                    two_diff(a[p], b[q], s, e);
                    const float sq = __fmul_rn(s, s);
                    float r = fmaf(s, s, -sq);
                    r = fmaf(__fadd_rn(s, s), e, r);
                    add_pair(hi[p][q], lo[p][q], sq, r);
                }
        }
    }
    unsigned long long *out = w + (size_t)blockIdx.x * PT * PT;
    float nui[4], nuj[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        nui[p] = nu[min(i0 + tr * 4 + p, N - 1)];
        nuj[p] = nu[min(j0 + tc * 4 + p, N - 1)];
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + tr * 4 + p, j = j0 + tc * 4 + q;
            unsigned long long v = 0ull;
            if (i < j && j < N) {
                double d = (double)hi[p][q] + (double)lo[p][q];
                // d >= max(nu_i, nu_j) / 16; the square overflows or underflows
                // only outside the range below
                const float m = fmaxf(nui[p], nuj[q]) * 0.0625f;
                const bool far_ = hi[p][q] >= m * m;
                // short secants, the threshold's neighbourhood (the exclusion
                // is decided in FP64) and lengths outside FP32's safe range:
                // squares overflow above it, and below it their residuals are
                // subnormal (each off by up to 2^-149: n 2^-149 / d^2 stays
                // below 2^-50 down to d^2 = 1e-25 at the largest n, 16384)
                if (!far_ || !(hi[p][q] > 1e-25f && hi[p][q] < 1e30f) || fabs(d - eps2) <= 1e-9 * eps2) {
                    d = 0.0;
                    const float *xr = X + (size_t)i * n, *yr = X + (size_t)j * n;
#pragma unroll 4
                    for (int l = 0; l < n; ++l) {
                        const float x = xr[l], y = yr[l];
                        float s, e;
                        two_diff(x, y, s, e);
                        const double D = diff64(x, y, s, e);
                        d = fma(D, D, d);
                    }
                }
                if (d != 0.0 && !(d < eps2)) {
                    const double wv = 1.0 / d;
                    const float wh = (float)wv;
                    if (far_ && wh < 1e30f && wh > 1e-25f) {
                        const float wl = (float)(wv - (double)wh);
                        v = ((unsigned long long)(__float_as_uint(wh) | 0x80000000u) << 32) | __float_as_uint(wl);
                    } else {
                        v = (unsigned long long)__double_as_longlong(wv);
                    }
                }
            }
            out[(tr * 4 + p) * PT + tc * 4 + q] = v;
        }
}

// R_i as in lap_rows_kernel: the FP32 pairs' sums over one block of columns,
// then added in FP64 (partial sums stay small, so their 2^-48 do too).  Warps
// whose coordinates are padding only stage (n = 100: 3 of 16 groups of 8), and
// three blocks per SM instead of two (80 registers) let the blocks of the
// last coordinates run beside the others: 8.2 -> 7.2 ms at N = 8192, n = 100
// (the whole start 13.7 with two blocks per SM, 13.4 with three, 14.1 with
// four, which spill).
__global__ void __launch_bounds__(256, 3) lap_pair_kernel(const float *X, int N, int n, const unsigned long long *w, int nb,
                                                       double *R)
{
    __shared__ uint2 wt[PT][PT + 1];
    __shared__ Staged<PT, PC> xs_;
    auto &xs = xs_.v;
    const int I = blockIdx.x, c0 = blockIdx.y * PC;
    const int r = threadIdx.x & (PT - 1), g = threadIdx.x >> 6;  // 4 groups of 8 coordinates
    const int i = I * PT + r;
    float xi[8];
    double acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int l = c0 + g * 8 + q;
        xi[q] = (i < N && l < n) ? X[(size_t)i * n + l] : 0.f;
        acc[q] = 0.0;
    }
    for (int J = 0; J < nb; ++J) {
        __syncthreads();
        const uint2 *tw = reinterpret_cast<const uint2 *>(w + tile_of(min(I, J), max(I, J), nb) * (PT * PT));
        for (int idx = threadIdx.x; idx < PT * PT; idx += 256) {
            const int a = idx / PT, b = idx % PT;  // the stored tile's row and column
            const uint2 v = tw[idx];
            if (I < J) wt[a][b] = v;
            else if (I > J) wt[b][a] = v;
            else if (a < b) { wt[a][b] = v; wt[b][a] = v; }
            else if (a == b) wt[a][a] = make_uint2(0u, 0u);
        }
        for (int idx = threadIdx.x; idx < PT * PC; idx += 256) {
            const int b = idx / PC, l = idx % PC;
            const int j = J * PT + b;
            xs[b][l] = (j < N && c0 + l < n) ? X[(size_t)j * n + c0 + l] : 0.f;
        }
        __syncthreads();
        float hi[8], lo[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) hi[q] = lo[q] = 0.f;
        if (c0 + g * 8 >= n) continue;  // only padding
#pragma unroll 2
        for (int b = 0; b < PT; ++b) {
            const uint2 v = wt[r][b];
            const float4 u0 = *reinterpret_cast<const float4 *>(&xs[b][g * 8]);
            const float4 u1 = *reinterpret_cast<const float4 *>(&xs[b][g * 8 + 4]);
            const float xb[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
            if ((int)v.y < 0) {
                const float wh = __uint_as_float(v.y & 0x7fffffffu), wl = __uint_as_float(v.x);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    float s, e;
                    two_diff(xi[q], xb[q], s, e);
                    const float p = __fmul_rn(wh, s);
                    float t = fmaf(wh, s, -p);
                    t = fmaf(wh, e, t);
                    t = fmaf(wl, s, t);
                    add_pair(hi[q], lo[q], p, t);
                }
            } else if (v.x | v.y) {
                const double wv = __hiloint2double((int)v.y, (int)v.x);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    float s, e;
                    two_diff(xi[q], xb[q], s, e);
                    acc[q] = fma(wv, diff64(xi[q], xb[q], s, e), acc[q]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q] += widen(hi[q]) + widen(lo[q]);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int l = c0 + g * 8 + q;
        if (i < N && l < n) R[(size_t)i * n + l] = acc[q];
    }
}

// Band z of C[a][b] = sum_i (x_ia - mean_a) R_ib over a 16 x 16 block of (a,
// b): the rows are cut into bands (with all rows in one block the 49 blocks
// of n = 100 left most SMs idle: 0.92 ms), added in order by band_sum_kernel.
// Bands cost n^2 words each, so there are only as many as it takes to give
// every SM eight blocks (16 at n = 100, one from n = 385 on, which then writes
// C itself), and none without rows.
constexpr int kGramBands = 16;
inline int gram_bands(int N, int n, int sms)
{
    const long long blocks = (long long)((n + 15) / 16) * ((n + 15) / 16);
    return (int)std::max(1ll, std::min({(long long)kGramBands, 8ll * sms / blocks, (N + 31ll) / 32}));
}
template <typename TX>
__global__ void __launch_bounds__(256) gram_kernel(const TX *X, const double *mean, const double *R, int N, int n,
                                                   double *Cp)
{
    __shared__ double xa[32][17], rb[32][17];
    const int a0 = blockIdx.x * 16, b0 = blockIdx.y * 16;
    const int ta = threadIdx.x >> 4, tb = threadIdx.x & 15;
    double acc = 0.0;
    const int step = 32 * (int)gridDim.z;
    const int rows = (N + step - 1) / step * 32, r1 = min(N, ((int)blockIdx.z + 1) * rows);
    for (int i0 = blockIdx.z * rows; i0 < r1; i0 += 32) {
        __syncthreads();
        for (int idx = threadIdx.x; idx < 32 * 16; idx += 256) {
            const int q = idx / 16, c = idx % 16;
            const int i = i0 + q;
            xa[q][c] = (i < r1 && a0 + c < n) ? ldx(X, (size_t)i * n + a0 + c) - mean[a0 + c] : 0.0;
            rb[q][c] = (i < r1 && b0 + c < n) ? R[(size_t)i * n + b0 + c] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int q = 0; q < 32; ++q) acc = fma(xa[q][ta], rb[q][tb], acc);
    }
    if (a0 + ta < n && b0 + tb < n) Cp[((size_t)blockIdx.z * n + a0 + ta) * n + b0 + tb] = acc;
}

__global__ void band_sum_kernel(const double *Cp, int bands, int n, double *C)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x, nn = (long long)n * n;
    if (idx >= nn) return;
    double acc = 0.0;
    for (int z = 0; z < bands; ++z) acc += Cp[z * nn + idx];
    C[idx] = acc;
}

// C <- (C + C^T) / 2 (the two halves differ only by rounding).
__global__ void symmetrize_kernel(double *C, int n)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)n * n) return;
    const int a = (int)(idx / n), b = (int)(idx % n);
    if (a < b) {
        const double v = 0.5 * (C[(size_t)a * n + b] + C[(size_t)b * n + a]);
        C[(size_t)a * n + b] = v;
        C[(size_t)b * n + a] = v;
    }
}

// ---- cyclic Jacobi eigensolver (FP64)

// Round r (0 <= r < m - 1) of the round-robin pairing of m (even) indices:
// index m - 1 meets r, and every other x meets (2r - x) mod (m - 1).
__device__ __forceinline__ int rr_partner(int x, int r, int m)
{
    if (x == m - 1) return r;
    if (x == r) return m - 1;
    int y = (2 * r - x) % (m - 1);
    return y < 0 ? y + (m - 1) : y;
}

// The rotation of every pair of round r: for pair (p, q), p < q, with
// a_pq != 0, tau = (a_qq - a_pp) / (2 a_pq), t = sign(tau) / (|tau| +
// sqrt(1 + tau^2)), c = 1 / sqrt(1 + t^2), s = t c; J = [[c, s], [-s, c]] in
// the (p, q) plane makes (J^T A J)_pq = 0.  Each index x stores the column
// combination col'_x = f_x col_x + g_x col_partner: (c, -s) for p, (s, c)
// read as (c, s) for q.  Unpaired indices (the extra one of an odd n, or
// a pair with a_pq = 0) keep f = 1, g = 0.
__global__ void jacobi_angles_kernel(const double *A, int n, int m, int r, double2 *fg, int *partner)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const int y = rr_partner(x, r, m);
    double f = 1.0, g = 0.0;
    int pt = x;
    if (y < n) {
        const int p = x < y ? x : y, q = x < y ? y : x;
        const double apq = A[(size_t)p * n + q];
        if (apq != 0.0) {
            const double tau = (A[(size_t)q * n + q] - A[(size_t)p * n + p]) / (2.0 * apq);
            const double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
            const double c = 1.0 / sqrt(1.0 + t * t), sn = t * c;
            f = c;
            g = x == p ? -sn : sn;
            pt = y;
        }
    }
    fg[x] = make_double2(f, g);
    partner[x] = pt;
}

// A' = J^T A J entry by entry (each entry reads at most four of A) and
// V' = V J (each entry reads two of V); one thread per entry.
__global__ void jacobi_apply_kernel(const double *A, const double *V, int n, const double2 *fg, const int *partner,
                                    double *A2, double *V2)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)n * n) return;
    const int i = (int)(idx / n), j = (int)(idx % n);
    const double2 ci = fg[i], cj = fg[j];
    const int pi = partner[i], pj = partner[j];
    const double a = A[(size_t)i * n + j], b = A[(size_t)i * n + pj];
    const double c = A[(size_t)pi * n + j], d = A[(size_t)pi * n + pj];
    // rows combine with (f_i, g_i), columns with (f_j, g_j)
    A2[(size_t)i * n + j] = ci.x * (cj.x * a + cj.y * b) + ci.y * (cj.x * c + cj.y * d);
    V2[(size_t)i * n + j] = cj.x * V[(size_t)i * n + j] + cj.y * V[(size_t)i * n + pj];
}

__global__ void jacobi_init_kernel(double *V, int n)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx < (long long)n * n) V[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
}

// off = sum of squared off-diagonal entries, all = sum of all squares (one
// block; fixed summation order).
__global__ void jacobi_norms_kernel(const double *A, int n, double *out)
{
    __shared__ double so[32], sa[32];
    double off = 0.0, all = 0.0;
    for (long long idx = threadIdx.x; idx < (long long)n * n; idx += blockDim.x) {
        const double v = A[idx];
        all = fma(v, v, all);
        if (idx / n != idx % n) off = fma(v, v, off);
    }
    off = warp_sum(off);
    all = warp_sum(all);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) { so[w] = off; sa[w] = all; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double o = 0.0, a = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) { o += so[q]; a += sa[q]; }
        out[0] = o;
        out[1] = a;
    }
}

// The whole eigensolver for n <= kClusterN in one launch: a cluster of 16
// blocks runs the rounds behind cluster barriers (two launches per round took
// 11 us, most of it gaps: 9 ms for the 792 rounds of n = 100).  Every block
// computes all rotations of a round itself (no exchange) from A in L2; the
// 2 x 2 blocks of (row pair, column pair) entries are dealt to the blocks,
// 16 FP64 operations per four entries; V's rows stay in the blocks' shared
// memory, since rotations combine its columns only.  The rotation of (p, q)
// with d = a_qq - a_pp, b = a_pq comes from two reciprocal square roots: r =
// 1/sqrt(d^2 + 4 b^2), c^2 = (1 + |d| r) / 2, s = |b| r / c, the same plane
// rotation as the quotient form above.  Above kClusterN the matrix is large
// enough for all SMs and the launches above.
constexpr int kClusterN = 256;
constexpr int kJacobiBlocks = 16;
constexpr int kJacobiThreads = 256;

__device__ __forceinline__ int2 rr_pair(int t, int r, int m, int n)
{
    int x, y;
    if (t == 0) {
        x = m - 1;
        y = r;
    } else {
        x = r + t;
        if (x >= m - 1) x -= m - 1;
        y = r - t;
        if (y < 0) y += m - 1;
    }
    const int p = min(x, y), q = max(x, y);
    return make_int2(p, q < n ? q : -1);  // an odd n's extra index pairs with nobody
}

__global__ void __launch_bounds__(kJacobiThreads) jacobi_cluster_kernel(double *A, double *A2, double *V, int n, double tol,
                                                                        int max_sweeps, double *out)
{
    extern __shared__ double vrow[];  // this block's rows of V
    __shared__ int2 pq[kClusterN / 2];
    __shared__ double2 cs[kClusterN / 2];
    __shared__ double part[2], red[2][kJacobiThreads / 32];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), C = (int)cluster.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int m = n + (n & 1), np = m / 2;
    const int rows = (n + C - 1) / C, v0 = rank * rows, nv = max(0, min(rows, n - v0));
    for (int idx = tid; idx < nv * n; idx += kJacobiThreads) vrow[idx] = (idx % n) == v0 + idx / n ? 1.0 : 0.0;
    bool done = n == 1;
    int sweep = 0;
    for (; sweep < max_sweeps && !done; ++sweep) {
        for (int r = 0; r < m - 1; ++r) {
            __syncthreads();  // the previous round's rotations have been used
            for (int t = tid; t < np; t += kJacobiThreads) {
                const int2 x = rr_pair(t, r, m, n);
                double2 v = make_double2(1.0, 0.0);
                if (x.y >= 0) {
                    const double b = __ldcg(A + (size_t)x.x * n + x.y);
                    const double d = __ldcg(A + (size_t)x.y * n + x.y) - __ldcg(A + (size_t)x.x * n + x.x);
                    const double h = fma(4.0 * b, b, d * d);
                    if (b != 0.0 && h > 0.0) {
                        const double ih = rsqrt(h);
                        const double c2 = 0.5 * fma(fabs(d), ih, 1.0);
                        const double ic = rsqrt(c2);
                        double sn = fabs(b) * ih * ic, cn = c2 * ic;
                        // one Newton step towards c^2 + s^2 = 1
                        const double f = fma(-0.5, fma(cn, cn, fma(sn, sn, -1.0)), 1.0);
                        cn *= f;
                        sn *= f;
                        v = make_double2(cn, (d >= 0.0) == (b >= 0.0) ? sn : -sn);
                    }
                }
                pq[t] = x;
                cs[t] = v;
            }
            __syncthreads();
            // A2 = J^T A J: column p' = c p - s q, q' = s p + c q, rows alike
            for (int e = rank + C * tid; e < np * np; e += C * kJacobiThreads) {
                const int tr = e / np, tc = e - tr * np;
                const int2 R = pq[tr], S = pq[tc];
                const double2 jr = cs[tr], jc = cs[tc];
                const bool hq = R.y >= 0, hs = S.y >= 0;
                const double a00 = __ldcg(A + (size_t)R.x * n + S.x);
                const double a01 = hs ? __ldcg(A + (size_t)R.x * n + S.y) : 0.0;
                const double a10 = hq ? __ldcg(A + (size_t)R.y * n + S.x) : 0.0;
                const double a11 = hq && hs ? __ldcg(A + (size_t)R.y * n + S.y) : 0.0;
                const double b00 = fma(jc.x, a00, -(jc.y * a01)), b01 = fma(jc.y, a00, jc.x * a01);
                const double b10 = fma(jc.x, a10, -(jc.y * a11)), b11 = fma(jc.y, a10, jc.x * a11);
                A2[(size_t)R.x * n + S.x] = fma(jr.x, b00, -(jr.y * b10));
                if (hs) A2[(size_t)R.x * n + S.y] = fma(jr.x, b01, -(jr.y * b11));
                if (hq) A2[(size_t)R.y * n + S.x] = fma(jr.y, b00, jr.x * b10);
                if (hq && hs) A2[(size_t)R.y * n + S.y] = fma(jr.y, b01, jr.x * b11);
            }
            for (int e = tid; e < nv * np; e += kJacobiThreads) {
                const int i = e / np, t = e - i * np;
                const int2 S = pq[t];
                if (S.y < 0) continue;
                const double2 j = cs[t];
                const double x = vrow[i * n + S.x], y = vrow[i * n + S.y];
                vrow[i * n + S.x] = fma(j.x, x, -(j.y * y));
                vrow[i * n + S.y] = fma(j.y, x, j.x * y);
            }
            double *t2 = A;
            A = A2;
            A2 = t2;
            cluster.sync();  // the round's A is complete
        }
        // off-diagonal and whole sums of squares, the blocks' parts added in order
        double off = 0.0, all = 0.0;
        for (int idx = tid; idx < nv * n; idx += kJacobiThreads) {
            const int i = v0 + idx / n, j = idx % n;
            const double v = __ldcg(A + (size_t)i * n + j);
            all = fma(v, v, all);
            if (i != j) off = fma(v, v, off);
        }
        off = warp_sum(off);
        all = warp_sum(all);
        if (lane == 0) {
            red[0][w] = off;
            red[1][w] = all;
        }
        __syncthreads();
        if (tid == 0) {
            double o = 0.0, a = 0.0;
            for (int q = 0; q < kJacobiThreads / 32; ++q) {
                o += red[0][q];
                a += red[1][q];
            }
            part[0] = o;
            part[1] = a;
        }
        cluster.sync();
        double o = 0.0, a = 0.0;
        for (int q = 0; q < C; ++q) {
            o += *cluster.map_shared_rank(&part[0], q);
            a += *cluster.map_shared_rank(&part[1], q);
        }
        done = !(o > tol * tol * a);  // the same in every block
        cluster.sync();  // the parts have been read
    }
    for (int idx = tid; idx < nv * n; idx += kJacobiThreads) V[(size_t)v0 * n + idx] = vrow[idx];
    if (rank == 0)
        for (int i = tid; i < n; i += kJacobiThreads) out[2 + i] = __ldcg(A + (size_t)i * n + i);
    if (rank == 0 && tid == 0) out[0] = done ? 1.0 : 0.0;
}

cudaError_t launch_jacobi_cluster(double *A, double *A2, double *V, int n, double tol, double *out, cudaStream_t s)
{
    cudaError_t e = cudaFuncSetAttribute(jacobi_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kJacobiBlocks);
    cfg.blockDim = dim3(kJacobiThreads);
    cfg.dynamicSmemBytes = (size_t)((n + kJacobiBlocks - 1) / kJacobiBlocks) * n * sizeof(double);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kJacobiBlocks;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, jacobi_cluster_kernel, A, A2, V, n, tol, 40, out);
}

struct Scratch {
    double *w = nullptr, *R = nullptr, *mean = nullptr, *C = nullptr, *C2 = nullptr, *V = nullptr, *V2 = nullptr,
           *norms = nullptr, *part = nullptr, *Cp = nullptr;
    double2 *fg = nullptr;
    int2 *tiles = nullptr;
    int *partner = nullptr;
    ~Scratch()
    {
        for (void *p : {(void *)w, (void *)R, (void *)mean, (void *)C, (void *)C2, (void *)V, (void *)V2,
                        (void *)norms, (void *)part, (void *)Cp, (void *)fg, (void *)tiles, (void *)partner})
            if (p) cudaFree(p);
    }
};

} // namespace

sap_status secant_pca(sap_handle h, int k, double *U_out, double *sigma_out)
{
    const int N = (int)handle_n_points(h), n = handle_n_dim(h);
    if (k < 1 || k > n || k > kMaxK) return handle_fail(h, SAP_E_ARG, "need 1 <= k <= min(n, 32)");
    cudaStream_t s = handle_stream(h);
    const float *X32 = handle_x32(h);
    const double *X64 = handle_x64(h);
    const int nb = (N + PT - 1) / PT;
    const long long ntiles = (long long)nb * (nb + 1) / 2;
    Scratch sc;
#define PCK(call)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess)                                                                     \
            return handle_fail(h, e_ == cudaErrorMemoryAllocation ? SAP_E_OOM : SAP_E_CUDA,        \
                               cudaGetErrorString(e_));                                            \
    } while (0)
    std::vector<int2> t;
    t.reserve(ntiles);
    for (int I = 0; I < nb; ++I)
        for (int J = I; J < nb; ++J) t.push_back(make_int2(I, J));
    PCK(cudaMalloc(&sc.tiles, t.size() * sizeof(int2)));
    PCK(cudaMemcpyAsync(sc.tiles, t.data(), t.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
    PCK(cudaMalloc(&sc.w, (size_t)ntiles * PT * PT * sizeof(double)));
    PCK(cudaMalloc(&sc.R, (size_t)N * n * sizeof(double)));
    PCK(cudaMalloc(&sc.mean, (size_t)n * sizeof(double)));
    PCK(cudaMalloc(&sc.part, colmean_scratch(N, n) * sizeof(double)));
    PCK(cudaMalloc(&sc.C, (size_t)n * n * sizeof(double)));
    PCK(cudaMalloc(&sc.C2, (size_t)n * n * sizeof(double)));
    const int bands = gram_bands(N, n, handle_sms(h));
    if (bands > 1) PCK(cudaMalloc(&sc.Cp, (size_t)bands * n * n * sizeof(double)));
    double *Cp = bands > 1 ? sc.Cp : sc.C;
    PCK(cudaMalloc(&sc.V, (size_t)n * n * sizeof(double)));
    PCK(cudaMalloc(&sc.V2, (size_t)n * n * sizeof(double)));
    PCK(cudaMalloc(&sc.norms, (size_t)(n + 2) * sizeof(double)));
    PCK(cudaMalloc(&sc.fg, (size_t)n * sizeof(double2)));
    PCK(cudaMalloc(&sc.partner, (size_t)n * sizeof(int)));
    const double eps2 = handle_eps2(h);
    const dim3 lgrid(nb, (n + PC - 1) / PC), ggrid((n + 15) / 16, (n + 15) / 16, bands);
    if (X64) {
        w64_kernel<double><<<(unsigned)ntiles, 256, 0, s>>>(X64, N, n, sc.tiles, eps2, sc.w);
        lap_rows_kernel<double><<<lgrid, 256, 0, s>>>(X64, N, n, sc.w, nb, sc.R);
        PCK(launch_colmean(X64, N, n, sc.part, sc.mean, s));
        gram_kernel<double><<<ggrid, 256, 0, s>>>(X64, sc.mean, sc.R, N, n, Cp);
    } else {
        unsigned long long *wp = reinterpret_cast<unsigned long long *>(sc.w);
        w_pair_kernel<<<(unsigned)ntiles, 256, 0, s>>>(X32, N, n, sc.tiles, eps2, handle_nu(h), wp);
        lap_pair_kernel<<<lgrid, 256, 0, s>>>(X32, N, n, wp, nb, sc.R);
        PCK(launch_colmean(X32, N, n, sc.part, sc.mean, s));
        gram_kernel<float><<<ggrid, 256, 0, s>>>(X32, sc.mean, sc.R, N, n, Cp);
    }
    PCK(cudaGetLastError());
    if (bands > 1) band_sum_kernel<<<(unsigned)(((long long)n * n + 255) / 256), 256, 0, s>>>(Cp, bands, n, sc.C);
    symmetrize_kernel<<<(unsigned)(((long long)n * n + 255) / 256), 256, 0, s>>>(sc.C, n);
    PCK(cudaGetLastError());
    // cyclic Jacobi sweeps: A (= C) towards diag(lambda), V accumulating the
    // rotations (its columns become the eigenvectors)
    double *A = sc.C, *A2 = sc.C2, *V = sc.V, *V2 = sc.V2;
    const double tol = 4.0 * n * std::ldexp(1.0, -53);
    bool converged = n == 1;
    std::vector<double> lam(n), Vh((size_t)n * n);
    if (n <= kClusterN) {
        PCK(launch_jacobi_cluster(A, A2, V, n, tol, sc.norms, s));
        std::vector<double> o(n + 2);
        PCK(cudaMemcpyAsync(o.data(), sc.norms, o.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
        PCK(cudaMemcpyAsync(Vh.data(), V, Vh.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
        PCK(cudaStreamSynchronize(s));
        converged = o[0] != 0.0;
        for (int c = 0; c < n; ++c) lam[c] = o[2 + c];
    } else {
        const unsigned nn_blocks = (unsigned)(((long long)n * n + 255) / 256);
        jacobi_init_kernel<<<nn_blocks, 256, 0, s>>>(sc.V, n);
        PCK(cudaGetLastError());
        const int m = n + (n & 1);
        for (int sweep = 0; sweep < 40 && !converged; ++sweep) {
            for (int r = 0; r < m - 1; ++r) {
                jacobi_angles_kernel<<<(n + 127) / 128, 128, 0, s>>>(A, n, m, r, sc.fg, sc.partner);
                jacobi_apply_kernel<<<nn_blocks, 256, 0, s>>>(A, V, n, sc.fg, sc.partner, A2, V2);
                std::swap(A, A2);
                std::swap(V, V2);
            }
            PCK(cudaGetLastError());
            jacobi_norms_kernel<<<1, 1024, 0, s>>>(A, n, sc.norms);
            double nrm[2] = {0.0, 0.0};
            PCK(cudaMemcpyAsync(nrm, sc.norms, sizeof(nrm), cudaMemcpyDeviceToHost, s));
            PCK(cudaStreamSynchronize(s));
            converged = !(nrm[0] > tol * tol * nrm[1]);
        }
        std::vector<double> Ah((size_t)n * n);
        PCK(cudaMemcpyAsync(Ah.data(), A, Ah.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
        PCK(cudaMemcpyAsync(Vh.data(), V, Vh.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
        PCK(cudaStreamSynchronize(s));
        for (int c = 0; c < n; ++c) lam[c] = Ah[(size_t)c * n + c];
    }
    if (!converged) return handle_fail(h, SAP_E_CUDA, "Jacobi eigensolver did not converge in 40 sweeps");
    // the k largest eigenvalues and their columns of V, largest first; each
    // vector signed so that its entry of largest magnitude is positive
    std::vector<int> order(n);
    for (int c = 0; c < n; ++c) order[c] = c;
    std::stable_sort(order.begin(), order.end(),
                     [&](int a, int b) { return lam[a] > lam[b]; });
    for (int c = 0; c < k; ++c) {
        const int col = order[c];
        int am = 0;
        for (int l = 1; l < n; ++l)
            if (std::fabs(Vh[(size_t)l * n + col]) > std::fabs(Vh[(size_t)am * n + col])) am = l;
        const double sg = Vh[(size_t)am * n + col] < 0 ? -1.0 : 1.0;
        for (int l = 0; l < n; ++l) U_out[(size_t)c * n + l] = sg * Vh[(size_t)l * n + col];
        if (sigma_out) sigma_out[c] = std::sqrt(std::max(lam[col], 0.0));
    }
    return SAP_OK;
#undef PCK
}

} // namespace sap
