// plain.cu -- the plain all-pairs pass: every unit secant is formed on the
// fly from tiles of X and projected with U (Sec. IV; the paper stores the
// secant matrix S, this form never materialises it).
//
// FP32 kernel: a block owns a 64 x 64 block of pairs (points i in block I,
// j in block J, I <= J; diagonal blocks keep i < j).  X rows of both blocks
// are staged in shared memory in chunks of 32 coordinates, transposed so a
// thread reads its 4 i's and 4 j's with one 16-byte load each; U's chunk is
// broadcast from shared memory as {u, u} pairs.  The next chunk is copied
// asynchronously while one is evaluated; chunk coordinate l of point r sits at
// [l][r ^ 4 (l % 8)] and a warp copies 8 coordinates (a 32-byte sector) of 4
// points, so neither side meets bank conflicts.  Bound by FP32 issue ((k + 2)
// n operations per pair): the arithmetic is packed FP32 pairs (two columns
// j), half the instructions with the same roundings in the same order.
// Each thread accumulates, for its 4 x 4 pairs,
//     d^2 = sum_l (x_il - x_jl)^2  and  z_c = sum_l u_lc (x_il - x_jl)
// with explicit FP32 differences and FMA chains, then r~ = sqrt(|z|^2 / d^2).
// Error model (u = 2^-24, gamma_m = m u/(1 - m u)):
//     |r~ - r| <= sqrt(k) gamma_{n+3} + (gamma_{n+2} + gamma_k + 3u) r,
// from |z~_c - z_c| <= gamma_{n+2} sum_l |u_lc||D_l| <= gamma_{n+2} ||D||.
// The block emits every pair that can still be the argmin under that model
// (see the selection scheme in sap_internal.cuh); pairs whose exclusion
// (d == 0, or d < eps of Sec. VII) is too close to call in FP32 are emitted
// for the FP64 tier to decide.
#include "sap_internal.cuh"
#include "tc_ptx.cuh"

namespace sap {
namespace {

constexpr int PB = 64;   // points per block edge
constexpr int LC = 32;   // coordinates per shared-memory chunk

template <int K>
__global__ void __launch_bounds__(256) plain_f32_kernel(PlainArgsF32 a)
{
    __shared__ __align__(16) float xsI[2][LC][PB];
    __shared__ __align__(16) float xsJ[2][LC][PB];
    __shared__ __align__(16) float us[2][LC][2 * K];
    __shared__ float red[32];
    __shared__ int scan[33];
    __shared__ int base_sh;

    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    // copies: chunk coordinate sl of the points sr, sr + 8, ...
    const int sl = ((tid >> 2) & 7) + 8 * ((tid >> 5) & 3), sr = (tid & 3) + 4 * (tid >> 7);

    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        const int2 IJ = a.tiles[t];
        const int i0 = IJ.x * PB, j0 = IJ.y * PB;
        uint64_t d2p[4][2];     // row p, columns 2 c and 2 c + 1
        uint64_t zp[4][2][K];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                d2p[p][c] = 0ull;
#pragma unroll
                for (int m = 0; m < K; ++m) zp[p][c][m] = 0ull;
            }
        auto copy = [&](int l0, int st) {
            const int gl = l0 + sl;
            const bool inl = gl < a.n;
#pragma unroll
            for (int q = 0; q < PB / 8; ++q) {
                const int r = sr + 8 * q, col = r ^ ((sl & 7) << 2);
                const bool ini = inl && i0 + r < a.N, inj = inl && j0 + r < a.N;
                tc::cp_async4(&xsI[st][sl][col], ini ? a.X + (size_t)(i0 + r) * a.n + gl : a.X, ini);
                tc::cp_async4(&xsJ[st][sl][col], inj ? a.X + (size_t)(j0 + r) * a.n + gl : a.X, inj);
            }
            for (int idx = tid; idx < LC * K * 2; idx += 256) {
                const int l = idx / (2 * K), c = (idx % (2 * K)) >> 1;
                const bool in = l0 + l < a.n;
                tc::cp_async4(&us[st][l][idx % (2 * K)], in ? a.U32 + (size_t)(l0 + l) * a.KP + c : a.U32, in);
            }
            tc::cp_async_commit();
        };
        __syncthreads();  // the previous tile's last chunk has been read
        copy(0, 0);
        for (int l0 = 0, st = 0; l0 < a.n; l0 += LC, st ^= 1) {
            if (l0 + LC < a.n) {
                copy(l0 + LC, st ^ 1);
                tc::cp_async_wait<1>();
            } else {
                tc::cp_async_wait<0>();
            }
            __syncthreads();
            const int lc = min(LC, a.n - l0);
#pragma unroll 4
            for (int l = 0; l < lc; ++l) {
                const int sw = (l & 7) << 2;
                const float4 xi = *reinterpret_cast<const float4 *>(&xsI[st][l][(ty * 4) ^ sw]);
                const ulonglong2 xj = *reinterpret_cast<const ulonglong2 *>(&xsJ[st][l][(tx * 4) ^ sw]);
                const float ai[4] = {xi.x, xi.y, xi.z, xi.w};
                uint64_t uu[K];
#pragma unroll
                for (int m = 0; m < K; ++m) uu[m] = *reinterpret_cast<const uint64_t *>(&us[st][l][2 * m]);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint64_t xx = tc::pk2(ai[p], ai[p]);
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const uint64_t D = tc::sub2(xx, c ? xj.y : xj.x);
                        d2p[p][c] = tc::fma2(D, D, d2p[p][c]);
#pragma unroll
                        for (int m = 0; m < K; ++m) zp[p][c][m] = tc::fma2(uu[m], D, zp[p][c][m]);
                    }
                }
            }
            __syncthreads();
        }
        float d2[4][4], z[4][4][K];
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float2 v = tc::upk2(d2p[p][c]);
                d2[p][2 * c] = v.x;
                d2[p][2 * c + 1] = v.y;
#pragma unroll
                for (int m = 0; m < K; ++m) {
                    const float2 y = tc::upk2(zp[p][c][m]);
                    z[p][2 * c][m] = y.x;
                    z[p][2 * c + 1][m] = y.y;
                }
            }

        // classify and evaluate the 16 pairs: 0 excluded, 1 normal, 2 decide in FP64
        float rt[4][4];
        int code[4][4];
        float mymin = INFINITY;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = i0 + ty * 4 + p, j = j0 + tx * 4 + q;
                const float dd = d2[p][q];
                int cd = 1;
                if (!(i < j && j < a.N)) cd = 0;
                else if (dd < 1e-30f) cd = 2;  // duplicate, or too short for FP32
                else if (a.eps2_hi > 0.f) {
                    if (dd < a.eps2_lo) cd = 0;
                    else if (dd < a.eps2_hi) cd = 2;
                }
                float zz = 0.f;
#pragma unroll
                for (int c = 0; c < K; ++c) zz = fmaf(z[p][q][c], z[p][q][c], zz);
                const float r = sqrtf(zz / dd);
                rt[p][q] = r;
                code[p][q] = cd;
                if (cd == 1) mymin = fminf(mymin, r);
            }

        const float bmin = block_min(mymin, red);
        float U = load_pos_float(&a.st->seed_ub);
        if (bmin < INFINITY) {
            const float ub = cert_upper(bmin, a.cert);
            if (tid == 0) atomic_min_pos_float(&a.st->run_ub1, ub);
            U = fminf(U, ub);
        }
        U = fminf(U, load_pos_float(&a.st->run_ub1));
        const float th = cert_emit_threshold(U, a.cert);

        int cnt = 0;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                cnt += (code[p][q] == 2 || (code[p][q] == 1 && rt[p][q] <= th)) ? 1 : 0;
        int total;
        int off = block_exclusive_scan(cnt, scan, &total);
        if (total == 0) continue;
        if (tid == 0) base_sh = (int)atomicAdd((unsigned int *)&a.st->cnt1, (unsigned int)total);
        __syncthreads();
        long long pos = (long long)(unsigned int)base_sh + off;
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (code[p][q] == 2 || (code[p][q] == 1 && rt[p][q] <= th)) {
                    if (pos < a.cand_cap)
                        a.cand[pos] = make_int2(i0 + ty * 4 + p, j0 + tx * 4 + q);
                    else
                        atomicOr(&a.st->status, ST_OVERFLOW);
                    ++pos;
                }
    }
}

// FP64 form (FP64 datasets): one thread per pair of a 16 x 16 block, X rows
// read through the cache.  The ratio is exact up to FP64 rounding; it is
// rounded to FP32 for the selection, hence the error model {0, 2^-23}.
// K is the basis width for k <= 8 (exactly k FP64 FMAs per coordinate:
// FP64 issue, not latency, is what a block of this kernel waits on), else
// kMaxK with the columns past k skipped.
template <int K>
__global__ void __launch_bounds__(256) plain_f64_kernel(PlainArgsF64 a)
{
    __shared__ float red[32];
    __shared__ int scan[33];
    __shared__ int base_sh;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    for (int t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        const int2 IJ = a.tiles[t];
        const int i = IJ.x * 16 + ty, j = IJ.y * 16 + tx;
        int cd = (i < j && j < a.N) ? 1 : 0;
        float rt = INFINITY;
        if (cd) {
            double d2 = 0.0;
            double z[K];
#pragma unroll
            for (int c = 0; c < K; ++c) z[c] = 0.0;
            const double *xi = a.X + (size_t)i * a.n;
            const double *xj = a.X + (size_t)j * a.n;
            for (int l = 0; l < a.n; ++l) {
                const double D = xi[l] - xj[l];
                d2 = fma(D, D, d2);
#pragma unroll
                for (int c = 0; c < K; ++c)
                    if (K <= 8 || c < a.k) z[c] = fma(a.U64[(size_t)c * a.n + l], D, z[c]);
            }
            if (d2 == 0.0 || d2 < a.eps2) {
                cd = 0;
            } else {
                double zz = 0.0;
#pragma unroll
                for (int c = 0; c < K; ++c)
                    if (K <= 8 || c < a.k) zz = fma(z[c], z[c], zz);
                rt = (float)sqrt(zz / d2);
            }
        }
        const float bmin = block_min(cd ? rt : INFINITY, red);
        float U = load_pos_float(&a.st->seed_ub);
        if (bmin < INFINITY) {
            const float ub = cert_upper(bmin, a.cert);
            if (tid == 0) atomic_min_pos_float(&a.st->run_ub1, ub);
            U = fminf(U, ub);
        }
        U = fminf(U, load_pos_float(&a.st->run_ub1));
        const float th = cert_emit_threshold(U, a.cert);
        const int emit = (cd && rt <= th) ? 1 : 0;
        int total;
        const int off = block_exclusive_scan(emit, scan, &total);
        if (total == 0) continue;
        if (tid == 0) base_sh = (int)atomicAdd((unsigned int *)&a.st->cnt1, (unsigned int)total);
        __syncthreads();
        if (emit) {
            const long long pos = (long long)(unsigned int)base_sh + off;
            if (pos < a.cand_cap) a.cand[pos] = make_int2(i, j);
            else atomicOr(&a.st->status, ST_OVERFLOW);
        }
    }
}

template <int K>
cudaError_t launch_k(const PlainArgsF32 &a, int grid, cudaStream_t s)
{
    plain_f32_kernel<K><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

} // namespace

cudaError_t launch_plain_f32(const PlainArgsF32 &a, cudaStream_t s)
{
    const int grid = a.grid;
    switch (a.k) {
#define SAP_CASE(KK) case KK: return launch_k<KK>(a, grid, s);
        SAP_CASE(1) SAP_CASE(2) SAP_CASE(3) SAP_CASE(4)
        SAP_CASE(5) SAP_CASE(6) SAP_CASE(7) SAP_CASE(8)
#undef SAP_CASE
    default:
        return cudaErrorInvalidValue;
    }
}

cudaError_t launch_plain_f64(const PlainArgsF64 &a, cudaStream_t s)
{
    switch (a.k) {
#define SAP_CASE(KK) case KK: plain_f64_kernel<KK><<<a.grid, 256, 0, s>>>(a); break;
        SAP_CASE(1) SAP_CASE(2) SAP_CASE(3) SAP_CASE(4)
        SAP_CASE(5) SAP_CASE(6) SAP_CASE(7) SAP_CASE(8)
#undef SAP_CASE
    default: plain_f64_kernel<kMaxK><<<a.grid, 256, 0, s>>>(a); break;
    }
    return cudaGetLastError();
}

} // namespace sap
