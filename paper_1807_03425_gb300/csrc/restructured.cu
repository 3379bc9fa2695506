// restructured.cu -- the restructured form of the SAP argmin step.
//
// For a basis U and Y = X U, U^T (x_i - x_j) = y_i - y_j, so
//     r_ij^2 = ||y_i - y_j||^2 * w_ij,   w_ij = 1 / ||x_i - x_j||^2.
// The lengths are computed once per dataset (and threshold eps, Sec. VII)
// from explicit FP32 differences; each iteration then costs one tensor-core
// product and one pass over the stored w (2 bytes per pair: BF16).
//
// Precision.  The rows of Y carry absolute errors of order eps_Y ||x - mean||
// (split-operand product, FP32 accumulation), so y_i - y_j cancels for close
// pairs.  Per pair the pass's error is bounded by
//     beta_ij = sqrt(k) eps_Y (nu_i + nu_j) / d_ij  (+ a relative FP32 term),
// with nu_i = ||x_i - mean||.  Pairs with beta_ij above a cap are "near": the
// pass skips them (w = NaN) and every iteration re-evaluates them from
// explicit differences instead.  All other pairs are certified to within the
// cap, so the pass emits every pair that can still be the argmin (selection
// scheme of sap_internal.cuh); a second tier narrows them and the FP64 tier
// decides (for n <= 256 and k <= 16 both inside the pass, restr_pass_kernel).
//
// Layout.  w is stored tile-major over the upper triangle: tile t = (I, J),
// I <= J, holds the 128 x 128 pairs (I*128 + a, J*128 + b) at t*128*128 --
// the FP32 w row-major, the BF16 w that the pass streams in groups of 8
// columns, the order its consumers read --; entries with i >= j, with an index beyond N, excluded pairs
// and near pairs hold NaN.
#include "restructured.cuh"
#include "colmean.cuh"
#include "tc_ptx.cuh"
#include "update_cluster.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

namespace sap {
namespace {

constexpr int T = kTile;       // 128
constexpr int WLC = 16;        // coordinates per chunk in the length prep

// ------------------------------------------------------------------ prep ---

__global__ void absmax_kernel(const float *X, size_t count, int n, const float *center,
                              unsigned int *out)
{
    float m = 0.f;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < count;
         idx += (size_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(X[idx] - center[idx % n]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

template <typename H>
__device__ __forceinline__ H to16(float v);
template <>
__device__ __forceinline__ __half to16<__half>(float v) { return __float2half_rn(v); }
template <>
__device__ __forceinline__ __nv_bfloat16 to16<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
__device__ __forceinline__ float from16(__half v) { return __half2float(v); }
__device__ __forceinline__ float from16(__nv_bfloat16 v) { return __bfloat162float(v); }

// hi = 16-bit(xs), lo = 16-bit((xs - hi) * lo_mul), xs = (x - mean) * scale;
// zero outside N x n.  The difference xs - hi is exact in FP32 and the
// scalings are powers of two.
template <typename H>
__global__ void split_kernel(const float *X, int N, int n, const float *center, float scale,
                             float lo_mul, H *hi, H *lo, int Npad, int NP)
{
    const size_t count = (size_t)Npad * NP;
    for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < count;
         idx += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(idx / NP), l = (int)(idx % NP);
        const float x = (r < N && l < n) ? X[(size_t)r * n + l] - center[l] : 0.f;
        const float xs = x * scale;
        const H h = to16<H>(xs);
        hi[idx] = h;
        lo[idx] = to16<H>((xs - from16(h)) * lo_mul);
    }
}

// nu_i = ||fl(x_i - mean)||_2, rounded up (one warp per row; 0 for pad rows).
__global__ void rownorm_kernel(const float *X, int N, int n, const float *center, float *nu, int Npad)
{
    const int row = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= Npad) return;
    double acc = 0.0;
    if (row < N)
        for (int l = lane; l < n; l += 32) {
            const double v = (double)(X[(size_t)row * n + l] - center[l]);
            acc = fma(v, v, acc);
        }
    acc = warp_sum(acc);
    if (lane == 0) nu[row] = row < N ? __double2float_ru(sqrt(acc)) * (1.0f + 1e-6f) : 0.f;
}

// ||x_i|| of the points as given (not centred), rounded up; 0 for pad rows.
__global__ void xnorm_kernel(const float *X, int N, int n, float *xn, int Npad)
{
    const int row = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (row >= Npad) return;
    double acc = 0.0;
    if (row < N)
        for (int l = lane; l < n; l += 32) {
            const double v = (double)X[(size_t)row * n + l];
            acc = fma(v, v, acc);
        }
    acc = warp_sum(acc);
    if (lane == 0) xn[row] = row < N ? __double2float_ru(sqrt(acc)) * (1.0f + 1e-6f) : 0.f;
}

struct WPrepArgs {
    const float *X;
    int N, n;
    const float *nu;
    const int2 *wtiles;
    float *w;
    __nv_bfloat16 *wb;       // BF16 1/d^2 of the stored pairs over yscale^2 (NaN elsewhere)
    float wb_scale;          // 1 / yscale^2 (a power of two)
    float eps2_lo, eps2_hi;  // FP32 window around eps^2 (0,0: no threshold)
    double eps2;
    float beta_coef;         // sqrt(k) * eps_Y, rounded up
    float b_cap;
    int2 *near;
    float *near_w;           // 1/d^2 of each near pair (+inf below FP32 range)
    unsigned int near_cap;
    unsigned int *counters;  // [0] near count, [1] excluded count (low), [2] status
};

// Exact decision in FP64 for pairs too close to call in FP32.
__device__ bool excluded_fp64(const float *X, int n, int i, int j, double eps2)
{
    double d2 = 0.0;
    for (int l = 0; l < n; ++l) {
        const double D = (double)X[(size_t)i * n + l] - (double)X[(size_t)j * n + l];
        d2 = fma(D, D, d2);
    }
    return d2 == 0.0 || d2 < eps2;
}

// One 128 x 128 tile of lengths per block: 256 threads, 8 x 8 pairs each.
// Bound by FP32 issue (2 n operations per pair; the 6 bytes per pair it
// writes take a tenth of that at n = 90), so the differences and squares are
// packed FP32 pairs (half the instructions, the same roundings in the same
// order) and the next chunk's points are copied asynchronously while a chunk
// is evaluated.  Chunk coordinate l of point r is staged at [l][r ^ 4 (l %
// 8)], and a warp copies 8 coordinates (one 32-byte sector) of 4 points: no
// bank conflicts on either side, and the readers' 16-byte groups stay whole.
__global__ void __launch_bounds__(256, 2) wprep_kernel(WPrepArgs a)
{
    __shared__ __align__(16) float xsI[2][WLC][T];
    __shared__ __align__(16) float xsJ[2][WLC][T];
    __shared__ int scan[33];
    __shared__ int base_sh;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int2 IJ = a.wtiles[blockIdx.x];
    const int i0 = IJ.x * T, j0 = IJ.y * T;
    uint64_t acc[8][4];  // row p, columns 2 c and 2 c + 1
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[p][c] = 0ull;
    // thread: chunk coordinate sl of the points sr, sr + 16, ...
    const int sl = ((tid >> 2) & 7) + 8 * ((tid >> 5) & 1), sr = (tid & 3) + 4 * (tid >> 6);
    auto copy = [&](int l0, int st) {
        const int gl = l0 + sl;
        const bool inl = gl < a.n;
#pragma unroll
        for (int q = 0; q < T / 16; ++q) {
            const int r = sr + 16 * q, col = r ^ ((sl & 7) << 2);
            const bool ini = inl && i0 + r < a.N, inj = inl && j0 + r < a.N;
            tc::cp_async4(&xsI[st][sl][col], ini ? a.X + (size_t)(i0 + r) * a.n + gl : a.X, ini);
            tc::cp_async4(&xsJ[st][sl][col], inj ? a.X + (size_t)(j0 + r) * a.n + gl : a.X, inj);
        }
        tc::cp_async_commit();
    };
    copy(0, 0);
    for (int l0 = 0, st = 0; l0 < a.n; l0 += WLC, st ^= 1) {
        if (l0 + WLC < a.n) {
            copy(l0 + WLC, st ^ 1);
            tc::cp_async_wait<1>();
        } else {
            tc::cp_async_wait<0>();
        }
        __syncthreads();
        // coordinates past n are zero on both sides: they add nothing
#pragma unroll 4
        for (int l = 0; l < WLC; ++l) {
            const int sw = (l & 7) << 2;
            const float4 ia = *reinterpret_cast<const float4 *>(&xsI[st][l][(ty * 8) ^ sw]);
            const float4 ib = *reinterpret_cast<const float4 *>(&xsI[st][l][(ty * 8 + 4) ^ sw]);
            const ulonglong2 ja = *reinterpret_cast<const ulonglong2 *>(&xsJ[st][l][(tx * 8) ^ sw]);
            const ulonglong2 jb = *reinterpret_cast<const ulonglong2 *>(&xsJ[st][l][(tx * 8 + 4) ^ sw]);
            const float xi[8] = {ia.x, ia.y, ia.z, ia.w, ib.x, ib.y, ib.z, ib.w};
            const uint64_t xj[4] = {ja.x, ja.y, jb.x, jb.y};
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                const uint64_t xx = tc::pk2(xi[p], xi[p]);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const uint64_t D = tc::sub2(xx, xj[c]);
                    acc[p][c] = tc::fma2(D, D, acc[p][c]);
                }
            }
        }
        __syncthreads();
    }
    float d2[8][8];
#pragma unroll
    for (int p = 0; p < 8; ++p)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float2 t = tc::upk2(acc[p][c]);
            d2[p][2 * c] = t.x;
            d2[p][2 * c + 1] = t.y;
        }
    float nuj[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) nuj[q] = __ldg(a.nu + j0 + tx * 8 + q);  // Npad entries
    const bool epson = a.eps2_hi > 0.f;
    int nnear = 0, nexcl = 0;
    unsigned long long near_bits = 0ull;  // bit p*8+q marks a near pair
    float *wt = a.w + (size_t)blockIdx.x * T * T;
    __nv_bfloat16 *ht = a.wb + (size_t)blockIdx.x * T * T;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        const int i = i0 + ty * 8 + p;
        const float nui = __ldg(a.nu + i);
        float out[8];
        __nv_bfloat16 hout[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int j = j0 + tx * 8 + q;
            const float dd = d2[p][q];
            float wv = __int_as_float(0x7fc00000);  // NaN: skipped by the pass
            __nv_bfloat16 hv = __ushort_as_bfloat16((unsigned short)0x7fc0);
            if (i < j && j < a.N) {
                int cls;  // 0 excluded, 1 near, 2 stored
                if (epson && dd < a.eps2_lo) cls = 0;
                else if ((epson && dd < a.eps2_hi) || dd < 1e-30f)
                    cls = excluded_fp64(a.X, a.n, i, j, a.eps2) ? 0 : 1;
                else {
                    const float inv = __frcp_rn(dd);
                    // the hardware estimate is within 2^-22 of 1/d: far
                    // inside the margin between the cap and the pass's bound
                    const float beta = a.beta_coef * (nui + nuj[q]) * rsqrtf(dd);
                    // near: the bound exceeds the cap
                    if (beta > a.b_cap) cls = 1;
                    else { cls = 2; wv = inv; hv = __float2bfloat16_rn(inv * a.wb_scale); }
                }
                if (cls == 0) ++nexcl;
                if (cls == 1) { ++nnear; near_bits |= 1ull << (p * 8 + q); }
            }
            out[q] = wv;
            hout[q] = hv;
        }
        float4 *dst = reinterpret_cast<float4 *>(wt + (size_t)(ty * 8 + p) * T + tx * 8);
        dst[0] = make_float4(out[0], out[1], out[2], out[3]);
        dst[1] = make_float4(out[4], out[5], out[6], out[7]);
        uint4 hp;
        hp.x = (unsigned)__bfloat16_as_ushort(hout[0]) | ((unsigned)__bfloat16_as_ushort(hout[1]) << 16);
        hp.y = (unsigned)__bfloat16_as_ushort(hout[2]) | ((unsigned)__bfloat16_as_ushort(hout[3]) << 16);
        hp.z = (unsigned)__bfloat16_as_ushort(hout[4]) | ((unsigned)__bfloat16_as_ushort(hout[5]) << 16);
        hp.w = (unsigned)__bfloat16_as_ushort(hout[6]) | ((unsigned)__bfloat16_as_ushort(hout[7]) << 16);
        *reinterpret_cast<uint4 *>(ht + ((size_t)tx * T + ty * 8 + p) * 8) = hp;  // column group tx, this row
    }
    int total;
    const int off = block_exclusive_scan(nnear, scan, &total);
    if (tid == 0 && total > 0) base_sh = (int)atomicAdd(&a.counters[0], (unsigned int)total);
    __syncthreads();
    if (total > 0) {
        unsigned int pos = (unsigned int)base_sh + off;
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (near_bits >> (p * 8 + q) & 1ull) {
                    if (pos < a.near_cap) {
                        a.near[pos] = make_int2(i0 + ty * 8 + p, j0 + tx * 8 + q);
                        a.near_w[pos] = d2[p][q] < 1e-30f ? INFINITY : 1.0f / d2[p][q];
                    } else {
                        atomicOr(&a.counters[2], 1u);
                    }
                    ++pos;
                }
    }
    int ex_total;
    block_exclusive_scan(nexcl, scan, &ex_total);
    if (tid == 0 && ex_total > 0)
        atomicAdd(reinterpret_cast<unsigned long long *>(&a.counters[4]), (unsigned long long)ex_total);
}

// ------------------------------------------------------- all-pairs pass ---

constexpr int kPassStagesMax = 5;

struct PassArgs {
    const uint16_t *wb;  // BF16 1/d^2 tiles over yscale^2 (tile-major upper triangle; NaN: skipped)
    const int2 *wtiles;
    int ntiles;
    const unsigned char *ops;  // this basis's A image in block 0 (gemm_tc.cuh: OpGroup)
    uint32_t ops_stride;       // bytes between blocks
    uint32_t img;              // bytes of one image
    int ksteps;                // MMA steps of 16
    int stage_y;               // 1: the FP32 Y of both sides is staged beside the tile
    float w_scale;             // yscale^2: a stored w times this is 1/d^2
    const float *Y;   // this basis's first component in block 0 of the block-major Y
    int Ykt;          // components per block of the Y buffer (block stride / 128)
    int Npad;
    const float *nu;  // ||fl(x_i - mean)||, rounded up (Npad)
    float beta;       // sqrt(k) eps_Y, rounded up: per-pair bound beta (nu_i + nu_j) / d_ij
    int stages;
    Cert cert;        // A = the cap of every stored pair's bound (b_cap), rho
    ProbState *st;
    int2 *cand;
    long long cap;
    int pdl;
    int k = 0;
    // second and third tiers inside the pass (non-null X; k <= 16): the
    // near pairs that Y cannot rule out and every emitted pair wait in their
    // warp's list; once its tiles are done, those that can still be the
    // argmin under the bound as it is then are evaluated, where many are left
    // first from explicit FP32 differences (the explicit tier's arithmetic
    // and error model, cert32), the survivors in FP64 (the FP64 recheck's
    // arithmetic).  Every block leaves its best (q = r^2, i, j) in partials[blockIdx.x] for the
    // update.  No list is written; st->cnt1 counts the emitted pairs,
    // st->cnt2 the FP64 evaluations.
    const float *X = nullptr;  // N x n FP32 points
    int N = 0, n = 0;
    const float *U32 = nullptr;  // n x KP FP32 basis (pad columns zero)
    int KP = 0;
    const double *U64 = nullptr;  // n x k FP64 basis, column-major
    double eps2 = 0.0;            // squared minimum secant length
    const int2 *near = nullptr;
    const float *near_w = nullptr;  // their 1/d^2 (+inf: too short for FP32)
    int n_near = 0;
    Partial *partials = nullptr;
    Cert cert32;
    // double-float tier (no X): the stored FP32 w narrows the emission, and
    // the near pairs that Y cannot rule out go to a list of their own
    const float *w32 = nullptr;   // FP32 1/d^2 tiles (row-major 128 x 128)
    int nb = 0;                   // point blocks per side
    long long tile0 = 0;          // global index of the first stored tile
    float rho32 = 0.f;            // relative error with the FP32 w
    int2 *near_out = nullptr;     // near_cap entries; st->cntn counts all
    int near_cap = 0;
};

// One ring stage: the BF16 1/d^2 tile (32 KB), the row block's A image and
// the column block's B image, the k components of both blocks' Y (when
// staged), then the 128 point norms nu of each side.
inline uint32_t pass_stage_bytes(int k, bool stage_y)
{
    return (uint32_t)T * T * 2 + 2u * op_image_bytes(k) + (stage_y ? 2u * k * T * 4 : 0u) + 2u * T * 4;
}

// Certified error of one stored pair's ratio from the tensor-core Y:
// |r~ - r| <= beta (nu_i + nu_j) / d_ij + rho r.  1/d_ij is taken as the
// square root of the stored BF16 w = 1/d^2 (relative error of w <= 2^-8, so
// of its root <= 2^-9 + 2^-23 with the FP32 root: inflated by 3 10^-3).  The
// same product the length preparation compares with b_cap.
__device__ __forceinline__ float sqrt_up(float x)  // the hardware square root (relative error 2^-22)
{
    float y;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float pair_bound(float beta, float nui, float nuj, float w)
{
    return beta * (nui + nuj) * sqrt_up(w) * 1.003f;
}

// Persistent, warp-specialised pass: one block per SM.  Each block's first
// `stages` tiles are blockIdx.x + it * gridDim.x (their constant parts are
// fetched before the previous kernel has finished); the remaining tiles
// follow the same stride, or with programmatic launch are handed out from a
// counter, so a block that starts late (its SM still busy with the previous
// kernels) takes fewer.  A producer warp keeps a ring of `stages`
// shared-memory buffers filled by 1-D TMA bulk copies, an MMA warp forms each
// tile's 128 x 128 products on the tensor cores (accumulator in tensor
// memory, two buffers), and 16 consumer warps read them back.  mbarriers hand
// the buffers over, so the loop has no block-wide barrier.
//
// Filter.  The contraction of the operand images (gemm_tc.cuh) is a certified
// lower bound of |y_i - y_j|^2 (in units of yscale), so its product with the
// stored w bounds r~^2 from below: a pair whose product exceeds the squared
// threshold cannot be the argmin, and a tile with no pair below it is done
// after one multiplication and one minimum per pair.  (A stored w is read as
// the upper half of a 32-bit word whose lower half is its neighbour: exact
// after a shift for the even columns, at most 2^-7 too large for the odd
// ones; kFilter widens the threshold by that.)  The rare tile that has one is
// re-evaluated where it matters from the FP32 rows of Y: r~^2 = |y_i - y_j|^2
// w, the value every bound below is certified for.
//
// What bounds it.  The differences and squares (2 k packed operations per
// pair of pairs) kept the FP32 pipe busy for 42 us per pass at N = 8192, k = 5
// and 184 us at N = 19939, k = 10; on the tensor cores they take 150-200
// cycles per tile, and what is left on the consumers (3 operations per pair)
// is below the stream of the stored lengths, about 1400 cycles per 32 KB tile
// and SM (6 TB/s).  Both passes now take 22 us and 82 us: the stream (12 and
// 70 us), 3 us until the first tile, 2-3 us for the survivors at the end.
//
// Bounds.  Every stored pair's error is at most b_p = beta (nu_i + nu_j) /
// d_ij <= A (= b_cap; pairs above it are on the near list).  The fast path
// tests each pair against the uniform A; a warp whose tile could tighten the
// upper bound takes the bound of its minimum from that pair's own b_p, and a
// pair that passes the uniform test is emitted only if it passes its own:
// r~_p <= U (1 + rho) + b_p.  Both refinements touch only the rare slow path.
constexpr int kConsumerWarps = 16;
constexpr int kPassThreads = (kConsumerWarps + 2) * 32;
constexpr int kTmemCols = 256;          // two 128-column accumulators
constexpr unsigned int kDense = 6;      // flagged columns per lane above which all 32 are evaluated
constexpr float kFilter = 1.0081f;      // (1 + 2^-7) (1 + 2.8e-4): odd columns' w, FP32 roundings

// A warp's pending pairs, packed with a lower bound of their ratio (pack_cand).
constexpr int kPending = 64;
constexpr int kQueue = 8;      // survivors the whole block evaluates together
// dynamic shared memory of the pass: the 227 KB a block may hold, less the
// static part (barriers, tile coordinates, the pending pairs)
constexpr int kPassDynSmem = 216 * 1024;

// Explicit FP32 differences of E pairs by one warp (lanes over the
// coordinates, the E (K + 1) sums reduced together), as in the explicit
// tier: lane e < E receives pair e's ratio rr and code (1: rr valid, 2:
// |x_i - x_j|^2 too small for FP32, a later tier decides; 0: none).
// expl32_finish reduces the per-lane sums acc[e (K + 1) + c].
template <int K, int E>
__device__ __forceinline__ void expl32_finish(float (&acc)[E * (K + 1)], const bool (&valid)[E], int lane, float &rr,
                                              int &code)
{
    constexpr int M = E * (K + 1);
    static_assert(M <= 32, "pairs per warp times components");
    constexpr int S = M <= 8 ? 8 : M <= 16 ? 16 : 32;
    constexpr int dup = 32 / S;
    float r[S];
#pragma unroll
    for (int q = 0; q < S; ++q) r[q] = q < M ? acc[q < M ? q : 0] : 0.f;
    const float t = warp_reduce_scatter<S>(r, lane);
    const int me = lane < E ? lane : 0;
    float z[K + 1];
#pragma unroll
    for (int c = 0; c <= K; ++c) z[c] = __shfl_sync(0xffffffffu, t, (me * (K + 1) + c) * dup);
    bool myvalid = valid[0];
#pragma unroll
    for (int e = 1; e < E; ++e)
        if (lane == e) myvalid = valid[e];
    const float dd = z[K];
    float zz = 0.f;
#pragma unroll
    for (int c = 0; c < K; ++c) zz = fmaf(z[c], z[c], zz);
    code = (lane >= E || !myvalid) ? 0 : (dd < 1e-30f ? 2 : 1);
    rr = code == 1 ? sqrtf(zz / dd) : INFINITY;
}

// One coordinate l of the sums: |D|^2 and U^T D for each pair's D[e]
template <int K, int E>
__device__ __forceinline__ void expl32_step(float (&acc)[E * (K + 1)], const float *U32, int KP, int l,
                                            const float (&D)[E])
{
    constexpr int KU = (K + 3) / 4 * 4;
    float u[KU];
#pragma unroll
    for (int c = 0; c < KU; c += 4) {
        // L2 only, like the point rows below: the pass leaves little L1
        // beside its shared memory (read-only loads through the L1 measured
        // 0.6-0.9 us slower per iteration)
        const float4 t = __ldcg(reinterpret_cast<const float4 *>(U32 + (size_t)l * KP + c));
        u[c] = t.x; u[c + 1] = t.y; u[c + 2] = t.z; u[c + 3] = t.w;
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
        acc[e * (K + 1) + K] = fmaf(D[e], D[e], acc[e * (K + 1) + K]);
#pragma unroll
        for (int c = 0; c < K; ++c) acc[e * (K + 1) + c] = fmaf(u[c], D[e], acc[e * (K + 1) + c]);
    }
}

template <int K, int E>
__device__ __forceinline__ void expl32_eval(const float *X, int n, const float *U32, int KP, const int2 (&pr)[E],
                                            const bool (&valid)[E], int lane, float &rr, int &code)
{
    float acc[E * (K + 1)];
#pragma unroll
    for (int q = 0; q < E * (K + 1); ++q) acc[q] = 0.f;
#pragma unroll 2
    for (int l = lane; l < n; l += 32) {
        float D[E];
#pragma unroll
        for (int e = 0; e < E; ++e) D[e] = __ldcg(X + (size_t)pr[e].x * n + l) - __ldcg(X + (size_t)pr[e].y * n + l);
        expl32_step<K, E>(acc, U32, KP, l, D);
    }
    expl32_finish<K, E>(acc, valid, lane, rr, code);
}

// K: compute width of the second tier inside the pass (EXPL); the filter and
// the FP32 re-evaluation take k at run time.
template <int K, bool EXPL>
__global__ void __launch_bounds__(kPassThreads, 1) restr_pass_kernel(const __grid_constant__ PassArgs a)
{
    // indexed directly (no integer round trip) so reads stay shared-memory loads
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t full[kPassStagesMax], empty[kPassStagesMax], tfull[2], tempty[2];
    __shared__ int2 sIJ[kPassStagesMax];
    __shared__ uint32_t tslot;
    __shared__ unsigned int sub;               // float bits: the block's best upper bound of the minimum
    __shared__ Partial pbest[kConsumerWarps];  // tiers inside: the warps' best pairs
    __shared__ unsigned long long pending[EXPL ? kConsumerWarps : 1][EXPL ? kPending : 1];
    __shared__ unsigned long long queue[EXPL ? kQueue : 1];  // the block's survivors
    __shared__ double entries[EXPL ? kQueue : 1][EXPL ? K + 1 : 1];
    __shared__ int nqueue;

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int S = a.stages, k = a.k;
    const uint32_t wbytes = T * T * 2, img = a.img, ybytes = a.stage_y ? (uint32_t)k * T * 4 : 0u;
    const uint32_t o_a = wbytes, o_b = o_a + img, o_yi = o_b + img, o_yj = o_yi + ybytes, o_nu = o_yj + ybytes;
    const uint32_t sbytes = o_nu + 2 * T * 4;
    // tiles below gridDim.x * S are static (it < S); the rest may be dynamic
    const int nall = blockIdx.x < (unsigned)a.ntiles ? (a.ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const int nstatic = nall < S ? nall : S;
    const long long budget = 4000000000ll;

    if (tid == 0) {
        sub = 0x7f800000u;
        nqueue = 0;
        for (int s = 0; s < S; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], kConsumerWarps);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&tfull[s], 1);
            tc::mbar_init(&tempty[s], kConsumerWarps);
        }
        tc::fence_mbar_init();
    }
    __syncthreads();
    // tensor memory, while the producer issues its first copies
    uint32_t tbase = 0;
    if (warp != kConsumerWarps) {
        if (warp == kConsumerWarps + 1) tc::tmem_alloc(&tslot, kTmemCols);
        tc::tc_fence_before();
        asm volatile("bar.sync 1, %0;" ::"n"(kPassThreads - 32) : "memory");
        tc::tc_fence_after();
        tbase = tslot;
    }

    if (warp == kConsumerWarps) {
        // ---------------- producer warp ----------------
        if (lane == 0) {
            // The stored lengths and point norms are constant: the first
            // stages' copies start before the product of this iteration has
            // finished (programmatic launch); Y follows after the wait.
            auto constant_part = [&](int s, int t, int2 IJ) {
                unsigned char *base = sm + (size_t)s * sbytes;
                tc::mbar_expect_tx(&full[s], sbytes);
                tc::bulk_g2s(base, a.wb + (size_t)t * T * T, wbytes, &full[s]);
                tc::bulk_g2s(base + o_nu, a.nu + (size_t)IJ.x * T, T * 4, &full[s]);
                tc::bulk_g2s(base + o_nu + T * 4, a.nu + (size_t)IJ.y * T, T * 4, &full[s]);
            };
            auto basis_part = [&](int s, int2 IJ) {
                unsigned char *base = sm + (size_t)s * sbytes;
                tc::bulk_g2s(base + o_a, a.ops + (size_t)IJ.x * a.ops_stride, img, &full[s]);
                tc::bulk_g2s(base + o_b, a.ops + (size_t)IJ.y * a.ops_stride + img, img, &full[s]);
                if (ybytes) {
                    tc::bulk_g2s(base + o_yi, a.Y + (size_t)IJ.x * a.Ykt * T, ybytes, &full[s]);
                    tc::bulk_g2s(base + o_yj, a.Y + (size_t)IJ.y * a.Ykt * T, ybytes, &full[s]);
                }
            };
            auto tile_at = [&](int t) {
                int2 IJ = a.wtiles[t];
                if (!SAP_BOUNDS_OK(a.st, IJ.x >= 0 && IJ.x <= IJ.y && IJ.y < a.Npad / T)) IJ = make_int2(0, 0);
                return IJ;
            };
            const int pre = nstatic;
            for (int it = 0; it < pre; ++it) {
                const int t = blockIdx.x + it * gridDim.x;
                const int2 IJ = tile_at(t);
                sIJ[it] = IJ;  // published by the mbarrier completion
                constant_part(it, t, IJ);
            }
            grid_dep_wait();
            grid_dep_launch();
            for (int it = 0; it < pre; ++it) basis_part(it, sIJ[it]);
            int issued = pre;
            bool marked = false;
            // Tiles after the first `stages`: with programmatic launch they
            // are claimed from a counter (some blocks start late); otherwise
            // block b takes b + it * gridDim.x.  Either way the next tile and
            // its coordinates are fetched one step ahead of their use.
            const int t0 = gridDim.x * S;
            auto next_tile = [&](int it) -> int {
                if (a.pdl) return t0 < a.ntiles ? t0 + (int)atomicAdd(&a.st->tile_next, 1u) : a.ntiles;
                return (int)blockIdx.x + it * (int)gridDim.x;
            };
            int tnext = next_tile(pre);
            int2 IJnext = tnext < a.ntiles ? tile_at(tnext) : make_int2(-1, -1);
            for (int it = pre;; ++it) {
                const int s = it % S;
                const int t = tnext;
                const int2 IJ = IJnext;
                if (t < a.ntiles) {
                    tnext = next_tile(it + 1);
                    IJnext = tnext < a.ntiles ? tile_at(tnext) : make_int2(-1, -1);
                }
                if (it >= S && !tc::mbar_wait_bounded(&empty[s], ((it / S) - 1) & 1, budget)) {
                    atomicOr(&a.st->status, ST_TIMEOUT);
                    break;
                }
                if (t >= a.ntiles) {
                    // no tile left: an arrival without bytes tells the others
                    sIJ[s] = make_int2(-1, -1);
                    tc::mbar_arrive(&full[s]);
                    marked = true;
                    break;
                }
                sIJ[s] = IJ;  // published by the mbarrier completion below
                constant_part(s, t, IJ);
                basis_part(s, IJ);
                ++issued;
            }
            // no copy of ours may still be in flight when the block exits
            // (the stage the end marker reused was consumed, so its copies
            // have landed; its barrier is past that phase)
            for (int it = issued > S ? issued - S : 0; it < issued; ++it)
                if (!(marked && it % S == issued % S)) tc::mbar_wait_bounded(&full[it % S], (it / S) & 1, budget);
        } else {
            grid_dep_wait();
            grid_dep_launch();
        }
        __syncwarp();
    } else if (warp == kConsumerWarps + 1) {
        // ---------------- MMA warp ----------------
        grid_dep_wait();
        grid_dep_launch();
        if (lane == 0) {
            const uint32_t idesc = tc::idesc_f16(T, T, 0);
            int it = 0;
            for (;; ++it) {
                const int s = it % S, buf = it & 1;
                if (!tc::mbar_wait_bounded(&full[s], (it / S) & 1, budget)) {
                    atomicOr(&a.st->status, ST_TIMEOUT);
                    break;
                }
                if (sIJ[s].x < 0) break;
                if (it >= 2 && !tc::mbar_wait_bounded(&tempty[buf], ((it >> 1) - 1) & 1, budget)) {
                    atomicOr(&a.st->status, ST_TIMEOUT);
                    break;
                }
                tc::tc_fence_after();
                const uint32_t sa = tc::smem_u32(sm + (size_t)s * sbytes + o_a);
                const uint32_t sb = sa + img;
                for (int q = 0; q < a.ksteps; ++q)
                    tc::mma_f16(tbase + buf * T, tc::desc_k_plain(sa + q * 4096, 2048, 128),
                                tc::desc_k_plain(sb + q * 4096, 2048, 128), idesc, q > 0 ? 1u : 0u);
                tc::mma_commit(&tfull[buf]);
            }
            // the tensor memory is freed below: no MMA may be in flight
            for (int j = it > 2 ? it - 2 : 0; j < it; ++j) tc::mbar_wait_bounded(&tfull[j & 1], (j >> 1) & 1, budget);
        }
        __syncwarp();
    } else {
    // ---------------- consumer warps ----------------
    // the lane's first near pair (constant over the run)
    const int nearG = (int)gridDim.x * kConsumerWarps, near0 = (int)blockIdx.x * kConsumerWarps + warp;
    int2 npr = make_int2(0, 0);
    float nw = INFINITY;
    if (near0 + lane * nearG < a.n_near) {
        npr = __ldcg(a.near + near0 + lane * nearG);
        nw = __ldcg(a.near_w + near0 + lane * nearG);
    }
    grid_dep_wait();  // Y, the bounds and the lists of this iteration
    grid_dep_launch();
    // this thread: row `row` of a tile, columns col0 .. col0 + 31
    const int row = 32 * (warp & 3) + lane, col0 = 32 * (warp >> 2);
    // Upper bounds of the minimum meet in shared memory; one warp per tile
    // exchanges the block's with the grid's (thousands of warps polling and
    // lowering one word cost 3 us at the start of a pass).
    if (lane == 0) atomicMin(&sub, __float_as_uint(load_pos_float(&a.st->seed_ub)));
    // r~ +- b_p to an upper and a lower bound (2 10^-6 for the roundings,
    // the hardware square root's 2^-22 among them)
    const float inv_up = 1.000002f / (1.0f - a.cert.rho), inv_dn = 0.999998f / (1.0f + a.cert.rho);
    auto bound_now = [&]() { return __uint_as_float(*(volatile unsigned int *)&sub); };
    auto lower_bound_to = [&](float ub) {
        if (lane == 0) atomicMin(&sub, __float_as_uint(ub));
    };
    // Second and FP64 tiers inside the pass.  A pair that Y cannot rule out
    // waits in the warp's pending list with a lower bound of its ratio; at the
    // end of the tiles (or when the list is full) those the bound of that
    // moment does not exclude are evaluated: two or fewer in FP64 at once,
    // more first from explicit FP32 differences, EX per round, which raises
    // their lower bounds and tightens the upper one.  Waiting matters: the
    // bound is loose while the first tiles are read, and an evaluation (2-5
    // us of latency) stalls the block's ring for pairs that are mostly
    // excluded a few tiles later (a look at the list after 6 tiles left the
    // slowest blocks 6 us behind at N = 8192 and 20 us at N = 12000).
    constexpr int EX = (K + 1) * 2 <= 32 ? 2 : 1;
    Partial best = {INFINITY, 0x7fffffff, 0x7fffffff};
    int nd = 0;  // pending pairs of this warp (warp-uniform)
    auto fp64_pair = [&](int2 ij) {
        if constexpr (EXPL) {
            if (!SAP_PAIR_OK(a.st, ij, a.N)) return;
            if (lane == 0) atomicAdd((unsigned int *)&a.st->cnt2, 1u);
            // the FP64 recheck's compute width for this k
            constexpr int KS = K <= 8 ? K : K <= 12 ? 12 : K <= 16 ? 16 : K <= 24 ? 24 : 32;
            double zz, d2;
            fp64_pair_parts<float, KS, true>(a.X, a.U64, a.n, a.k, ij, lane, zz, d2);
            if (d2 == 0.0 || d2 < a.eps2) return;
            const double q = zz / d2;
            if (better_q(q, ij.x, ij.y, best.r, best.i, best.j)) best = Partial{q, ij.x, ij.y};
        }
    };
    auto flush = [&]() {
        if constexpr (EXPL) {
            __syncwarp();
            unsigned long long *list = pending[warp];
            // one bit per pending pair that can still be the argmin
            auto alive = [&](unsigned int (&m)[2]) {
                const float th = bound_now() * 1.000001f;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int q = 32 * h + lane;
                    m[h] = __ballot_sync(0xffffffffu, q < nd && packed_ratio(list[q < nd ? q : 0]) <= th);
                }
            };
            auto take = [](unsigned int (&m)[2]) {  // the lowest set bit, removed
                const int h = m[0] ? 0 : 1, e = __ffs(m[h]) - 1;
                m[h] &= m[h] - 1u;
                return 32 * h + e;
            };
            unsigned int m[2];
            alive(m);
            if (__popc(m[0]) + __popc(m[1]) > 2) {
                unsigned int rem[2] = {m[0], m[1]};
                while (rem[0] | rem[1]) {
                    int2 pr[EX];
                    int at[EX];
                    bool valid[EX];
#pragma unroll
                    for (int e = 0; e < EX; ++e) {
                        valid[e] = (rem[0] | rem[1]) != 0u;
                        at[e] = valid[e] ? take(rem) : 0;
                        pr[e] = valid[e] ? packed_pair(list[at[e]]) : make_int2(0, 0);
                    }
                    float rr;
                    int code;
                    expl32_eval<K, EX>(a.X, a.n, a.U32, a.KP, pr, valid, lane, rr, code);
                    const float wmin = warp_min(rr);
                    if (wmin < INFINITY) {
                        const float ub = cert_upper(wmin, a.cert32);
                        if (ub < bound_now()) {
                            lower_bound_to(ub);
                            if (lane == 0) atomic_min_pos_float(&a.st->run_ub1, ub);
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int e = 0; e < EX; ++e)
                        if (lane == e && valid[e])
                            list[at[e]] = pack_cand(pr[e].x, pr[e].y,
                                                    fmaxf((rr - a.cert32.A) / (1.0f + a.cert32.rho) * 0.999998f, 0.f),
                                                    code == 2);
                    __syncwarp();
                }
                alive(m);
            }
            while (m[0] | m[1]) fp64_pair(packed_pair(list[take(m)]));
            __syncwarp();
            nd = 0;
        }
    };
    // the pairs of the lanes with keep set join the list
    auto append = [&](int pi, int pj, float lo, bool keep) {
        if constexpr (EXPL) {
            const unsigned int m = __ballot_sync(0xffffffffu, keep);
            const int c = __popc(m);
            if (c == 0) return;
            if (nd + c > kPending) flush();
            if (keep) pending[warp][nd + __popc(m & ((1u << lane) - 1u))] = pack_cand(pi, pj, lo, false);
            nd += c;
        }
    };
    // The near pairs, one per lane: their ratio from Y with their own (large)
    // bound rules most of them out in O(k); it also bounds the minimum.
    auto near_pairs = [&]() {
        {
            for (long long base = 0; base < a.n_near; base += 32ll * nearG) {
                const long long idx = base + near0 + (long long)lane * nearG;
                int2 pr = npr;
                float ub = INFINITY, lo = INFINITY;
                if (idx < a.n_near) {
                    if (base > 0) {
                        pr = __ldcg(a.near + idx);
                        nw = __ldcg(a.near_w + idx);
                    }
                    if (SAP_PAIR_OK(a.st, pr, a.N)) {
                        const float *yi = a.Y + (size_t)(pr.x >> 7) * a.Ykt * T + (pr.x & (T - 1));
                        const float *yj = a.Y + (size_t)(pr.y >> 7) * a.Ykt * T + (pr.y & (T - 1));
                        float zz = 0.f;
                        if constexpr (EXPL) {
#pragma unroll
                            for (int c = 0; c < K; ++c)
                                if (c < k) {
                                    const float e = __ldcg(yi + c * T) - __ldcg(yj + c * T);
                                    zz = fmaf(e, e, zz);
                                }
                        } else {
#pragma unroll 8
                            for (int c = 0; c < k; ++c) {
                                const float e = __ldcg(yi + c * T) - __ldcg(yj + c * T);
                                zz = fmaf(e, e, zz);
                            }
                        }
                        if (nw < INFINITY) {
                            const float r = sqrt_up(zz * nw);
                            const float b = pair_bound(a.beta, __ldg(a.nu + pr.x), __ldg(a.nu + pr.y), nw);
                            ub = (r + b) * inv_up;
                            lo = fmaxf((r - b) * inv_dn, 0.f);
                        } else {
                            lo = 0.f;  // too short for FP32: a later tier decides
                        }
                    }
                }
                ub = warp_min(ub);
                const float U = bound_now();
                if (ub < U) lower_bound_to(ub);
                const bool keep = lo <= fminf(U, ub) * 1.000001f && lo < INFINITY;
                if constexpr (EXPL) {
                    append(pr.x, pr.y, lo, keep);
                } else {
                    const unsigned int m = __ballot_sync(0xffffffffu, keep);
                    if (!m) continue;
                    unsigned int at = 0;
                    if (lane == 0) at = atomicAdd((unsigned int *)&a.st->cntn, (unsigned int)__popc(m));
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
                    if (keep && at < (unsigned int)a.near_cap) a.near_out[at] = pr;
                }
            }
        }
    };
    if (EXPL) near_pairs();  // while the first stages' copies land
    // ring position and barrier phases, advanced without integer division
    int s = 0;
    uint32_t phase = 0;
    const uint32_t taddr = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + col0;
    const float wsc = a.w_scale;
    for (int it = 0;; ++it, s = (s + 1 == S) ? 0 : s + 1, phase ^= (s == 0) ? 1u : 0u) {
        if (!__all_sync(0xffffffffu, tc::mbar_wait_bounded(&full[s], phase, budget))) {
            if (lane == 0) atomicOr(&a.st->status, ST_TIMEOUT);
            break;
        }
        const int2 IJ = sIJ[s];
        if (IJ.x < 0) break;  // the producer has no more tiles
        const bool exch = warp == (it & (kConsumerWarps - 1));
        float gnow = INFINITY;
        if (exch) gnow = load_pos_float(&a.st->run_ub1);  // consumed after the tile
        const unsigned char *stage = sm + (size_t)s * sbytes;
        const int buf = it & 1;
        if (!__all_sync(0xffffffffu, tc::mbar_wait_bounded(&tfull[buf], (it >> 1) & 1, budget))) {
            if (lane == 0) atomicOr(&a.st->status, ST_TIMEOUT);
            break;
        }
        tc::tc_fence_after();
        float v[32];  // lower bounds of |y_i - y_j|^2, then of r~^2
        tc::tmem_ld32(taddr + buf * T, v);
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&tempty[buf]);
        float m0 = INFINITY, m1 = INFINITY;
        {
            const uint4 *wp = reinterpret_cast<const uint4 *>(stage) + (col0 >> 3) * T + row;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint4 w4 = wp[c * T];
                const uint32_t ww[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int e = c * 8 + 2 * q;
                    const uint64_t p = tc::mul2(tc::pk2(v[e], v[e + 1]),
                                                tc::pk2(__uint_as_float(ww[q] << 16), __uint_as_float(ww[q])));
                    const float2 t = tc::upk2(p);
                    v[e] = t.x;
                    v[e + 1] = t.y;
                    m0 = fminf(m0, t.x);
                    m1 = fminf(m1, t.y);
                }
            }
        }
        const float mymin = fminf(m0, m1);
        if (exch) {
            const float mine = bound_now();
            if (gnow < mine) lower_bound_to(gnow);
            else if (mine < gnow && lane == 0) atomic_min_pos_float(&a.st->run_ub1, mine);
        }
        float U = fminf(gnow, bound_now());
        float thc = cert_emit_threshold(U, a.cert);
        float thc2 = thc * thc * 1.000001f;
        // thc >= U, so a tile that could tighten the bound (minimum below
        // U^2) also fails this test: the fast path needs no warp minimum
        if (!__any_sync(0xffffffffu, mymin <= thc2 * kFilter)) {
            // fast path: nothing in this tile can bound or be the minimum
            if (lane == 0) tc::mbar_arrive(&empty[s]);
            continue;
        }
        // ---- slow path: FP32 rows of Y
        const float *sI = reinterpret_cast<const float *>(stage + o_yi), *sJ = reinterpret_cast<const float *>(stage + o_yj);
        const float *gI = a.Y + (size_t)IJ.x * a.Ykt * T, *gJ = a.Y + (size_t)IJ.y * a.Ykt * T;
        const uint16_t *hs = reinterpret_cast<const uint16_t *>(stage);
        const float *nuI = reinterpret_cast<const float *>(stage + o_nu), *nuJ = nuI + T;
        const float *w32t = nullptr;  // the tile's FP32 w
        if (!EXPL && a.w32)
            w32t = a.w32 + ((long long)IJ.x * a.nb - (long long)IJ.x * (IJ.x - 1) / 2 + (IJ.y - IJ.x) - a.tile0) * (T * T);
        // r~^2 of pair (r, c), its w in w
        auto pair_q = [&](int r, int c, float &w) {
            w = __uint_as_float((uint32_t)hs[((c >> 3) * T + r) * 8 + (c & 7)] << 16) * wsc;
            float q = 0.f;
            if constexpr (EXPL && K <= 12) {  // staged (pass_stages_y)
#pragma unroll
                for (int m = 0; m < K; ++m)
                    if (m < k) {
                        const float e = sI[m * T + r] - sJ[m * T + c];
                        q = fmaf(e, e, q);
                    }
            } else if (ybytes) {
                for (int m = 0; m < k; ++m) {
                    const float e = sI[m * T + r] - sJ[m * T + c];
                    q = fmaf(e, e, q);
                }
            } else {
#pragma unroll 4
                for (int m = 0; m < k; ++m) {
                    const float e = __ldcg(gI + m * T + r) - __ldcg(gJ + m * T + c);
                    q = fmaf(e, e, q);
                }
            }
            return q * w;
        };
        const float wmin = warp_min(mymin);
        if (wmin < INFINITY) {
            // the bound of (about) the tile's minimum from that pair's own error
            const int src = __ffs(__ballot_sync(0xffffffffu, mymin == wmin)) - 1;
            float ub = INFINITY;
            if (lane == src) {
                int pcol = col0;
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    if (v[e] == wmin) pcol = col0 + e;
                float w;
                const float r = sqrt_up(pair_q(row, pcol, w));
                if (r < U) ub = (r + pair_bound(a.beta, nuI[row], nuJ[pcol], w)) * inv_up;
                if (!EXPL && w32t && ub < INFINITY) {
                    const float w32 = __ldg(w32t + row * T + pcol);
                    ub = fminf(ub, (r * sqrt_up(w32 / w) + pair_bound(a.beta, nuI[row], nuJ[pcol], w)) *
                                       (1.000003f / (1.0f - a.rho32)));
                }
            }
            ub = __shfl_sync(0xffffffffu, ub, src);
            if (ub < U) {
                lower_bound_to(ub);
                U = ub;
                thc = cert_emit_threshold(U, a.cert);
                thc2 = thc * thc * 1.000001f;
            }
        }
        uint32_t flag = 0u, emit = 0u;
        if (mymin <= thc2 * kFilter)
#pragma unroll
            for (int e = 0; e < 32; ++e)
                if (v[e] <= thc2 * kFilter) flag |= 1u << e;
        // Where the filter tells little (its error is relative to the points'
        // distances from the mean, and absolute at the scale of the farthest
        // one: a point far out leaves most pairs flagged, and the lowest bound
        // says nothing about where the minimum is) the lane's 32 columns are
        // evaluated eight at a time instead of a pair per lane and turn, with
        // pair_q's operations, and the true minimum tightens the bound (once
        // more if that still leaves many).  Per iteration, with one point
        // 10^4 times farther out: 4116 -> 174 us at N = 3000, n = 100, k = 20
        // (109 without the point), 158 -> 82 at N = 8192, k = 5 (41), 141 ->
        // 73 at N = 3000, n = 300, k = 6 (63).  From 7 flagged columns in a
        // lane on: with 13 and 21 the same took 171 and 187, 86 and 94, 70
        // and 71 us, and with noise at k = 5 (58) 83 and 96.
        bool many = __reduce_max_sync(0xffffffffu, (unsigned int)__popc(flag)) > kDense;
        if (many) {
            // The lanes read the bound each for itself and other warps lower
            // it meanwhile, so it may differ between them.  What follows
            // leaves its loop by comparisons with it and meets in warp-wide
            // operations: one value for the warp (any lane's is valid).
            U = __shfl_sync(0xffffffffu, U, 0);
            thc = cert_emit_threshold(U, a.cert);
            thc2 = thc * thc * 1.000001f;
        }
        for (int rep = 0; rep < 2 && many; ++rep) {
            const bool staged = (EXPL && K <= 12) || ybytes;  // (pass_stages_y)
            const float *yI = staged ? sI : gI, *yJ = staged ? sJ : gJ;
            float mn = INFINITY;
            int mc = col0;
            flag = 0u;
#pragma unroll 1
            for (int c = 0; c < 32; c += 8) {
                uint64_t q2[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll 4
                for (int m = 0; m < k; ++m) {
                    const float yi = staged ? yI[m * T + row] : __ldcg(yI + m * T + row);
                    const ulonglong2 *g = reinterpret_cast<const ulonglong2 *>(yJ + m * T + col0 + c);
                    const ulonglong2 ya = staged ? g[0] : __ldcg(g), yb = staged ? g[1] : __ldcg(g + 1);
                    const uint64_t yy = tc::pk2(yi, yi);
                    const uint64_t d0 = tc::sub2(yy, ya.x), d1 = tc::sub2(yy, ya.y);
                    const uint64_t d2 = tc::sub2(yy, yb.x), d3 = tc::sub2(yy, yb.y);
                    q2[0] = tc::fma2(d0, d0, q2[0]);
                    q2[1] = tc::fma2(d1, d1, q2[1]);
                    q2[2] = tc::fma2(d2, d2, q2[2]);
                    q2[3] = tc::fma2(d3, d3, q2[3]);
                }
                const uint4 w4 = *(reinterpret_cast<const uint4 *>(stage) + ((col0 + c) >> 3) * T + row);
                const uint32_t ww[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float2 t = tc::upk2(q2[e >> 1]);
                    const float w = __uint_as_float((e & 1) ? ww[e >> 1] & 0xffff0000u : ww[e >> 1] << 16) * wsc;
                    const float q = ((e & 1) ? t.y : t.x) * w;
                    if (q < mn) {
                        mn = q;
                        mc = col0 + c + e;
                    }
                    if (q <= thc2) flag |= 1u << (c + e);
                }
            }
            const float qmin = warp_min(mn);
            if (!(qmin <= thc2)) break;
            const int src = __ffs(__ballot_sync(0xffffffffu, mn == qmin)) - 1;
            float ub = INFINITY;
            if (lane == src) {
                const float w = __uint_as_float((uint32_t)hs[((mc >> 3) * T + row) * 8 + (mc & 7)] << 16) * wsc;
                const float r = sqrt_up(qmin);
                if (r < U) ub = (r + pair_bound(a.beta, nuI[row], nuJ[mc], w)) * inv_up;
            }
            ub = __shfl_sync(0xffffffffu, ub, src);
            if (!(ub < U)) break;
            lower_bound_to(ub);
            U = ub;
            thc = cert_emit_threshold(U, a.cert);
            thc2 = thc * thc * 1.000001f;
            many = __reduce_max_sync(0xffffffffu, (unsigned int)__popc(flag)) > kDense;
        }
        // emission: the uniform test, then each survivor against its own bound
        const float ut = U * (1.0f + a.cert.rho);
        const int i0 = IJ.x * T, j0 = IJ.y * T;
        if constexpr (EXPL) {
            int total = 0;
            while (__any_sync(0xffffffffu, flag != 0u)) {  // one flagged pair per lane
                bool keep = false;
                float lo = 0.f;
                const int e = flag ? __ffs(flag) - 1 : 0;
                if (flag) {
                    float w;
                    const float q = pair_q(row, col0 + e, w);
                    if (q <= thc2) {
                        const float bp = pair_bound(a.beta, nuI[row], nuJ[col0 + e], w);
                        const float th = (ut + bp) * 1.000001f;
                        keep = q <= th * th * 1.000001f;
                        lo = fmaxf((sqrt_up(q) - bp) * inv_dn, 0.f);
                    }
                    flag &= flag - 1u;
                }
                total += __popc(__ballot_sync(0xffffffffu, keep));
                append(i0 + row, j0 + col0 + e, lo, keep);
            }
            // the warp's reads of stage s are done
            __syncwarp();
            if (lane == 0) {
                tc::mbar_arrive(&empty[s]);
                if (total) atomicAdd((unsigned int *)&a.st->cnt1, (unsigned int)total);
            }
        } else {
            while (flag) {
                const int e = __ffs(flag) - 1;
                flag &= flag - 1u;
                float w;
                float q = pair_q(row, col0 + e, w);
                if (q <= thc2) {
                    const float bp = pair_bound(a.beta, nuI[row], nuJ[col0 + e], w);
                    float th = (ut + bp) * 1.000001f;
                    if (q > th * th * 1.000001f) continue;
                    if (w32t) {
                        // the FP32 w: an eighth of the BF16 rounding's window
                        q = q / w * __ldg(w32t + row * T + col0 + e);
                        th = (U * (1.0f + a.rho32) + bp) * 1.000002f;
                        if (q > th * th * 1.000001f) continue;
                    }
                    emit |= 1u << e;
                }
            }
            const int cnt = __popc(emit);
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&empty[s]);
            const int total = __reduce_add_sync(0xffffffffu, cnt);
            if (total == 0) continue;
            unsigned int cbase = 0;
            if (lane == 0) cbase = atomicAdd((unsigned int *)&a.st->cnt1, (unsigned int)total);
            int incl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            long long pos = (long long)__shfl_sync(0xffffffffu, cbase, 0) + incl - cnt;
            while (emit) {
                const int e = __ffs(emit) - 1;
                emit &= emit - 1u;
                if (pos < a.cap) a.cand[pos] = make_int2(i0 + row, j0 + col0 + e);
                else atomicOr(&a.st->status, ST_OVERFLOW);
                ++pos;
            }
        }
    }
    if constexpr (!EXPL) {
        if (a.n_near > 0) {
            // the near pairs against the grid's bound, now tight
            if (lane == 0) atomicMin(&sub, __float_as_uint(load_pos_float(&a.st->run_ub1)));
            __syncwarp();
            near_pairs();
            if (lane == 0) atomic_min_pos_float(&a.st->run_ub1, bound_now());
        }
    }
    if constexpr (EXPL) {
        // The pending pairs against the grid's bound.  Usually one or two
        // pairs of the whole grid survive: the block evaluates its own
        // together, one warp per entry of U^T D and |D|^2 (a warp alone
        // needs 5-8 us for one pair, most of it FP64 issue).
        auto meet = [&]() { asm volatile("bar.sync 2, %0;" ::"n"(kConsumerWarps * 32) : "memory"); };
        // the usual sizes: warp c holds entry c's basis column in registers,
        // loaded ahead of the barriers that follow
        const bool direct = a.n <= kSliceN && k < kConsumerWarps;
        double ur[kSliceN / 32];
        if (direct && warp < k)
#pragma unroll
            for (int t = 0; t < kSliceN / 32; ++t)
                ur[t] = lane + 32 * t < a.n ? __ldcg(a.U64 + (size_t)warp * a.n + lane + 32 * t) : 0.0;
        meet();
        if (warp == 0 && lane == 0) {
            const float g = load_pos_float(&a.st->run_ub1), mine = bound_now();
            if (mine < g) atomic_min_pos_float(&a.st->run_ub1, mine);
            else lower_bound_to(g);
        }
        meet();
        {
            const float th = bound_now() * 1.000001f;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q = 32 * h + lane;
                if (q < nd && packed_ratio(pending[warp][q]) <= th) {
                    const int at = atomicAdd(&nqueue, 1);
                    if (at < kQueue) queue[at] = pending[warp][q];
                }
            }
        }
        meet();
        const int nq = nqueue;
        if (nq > kQueue || (size_t)nq * a.n * sizeof(double) > (size_t)T * T * 2) {
            flush();
        } else if (nq > 0) {
            // D of every survivor, in the first ring stage (its tiles are done)
            double *Ds = reinterpret_cast<double *>(sm);
            for (int t = tid; t < nq * a.n; t += kConsumerWarps * 32) {
                const int q = t / a.n, l = t - q * a.n;
                const int2 ij = packed_pair(queue[q]);
                Ds[t] = SAP_PAIR_OK(a.st, ij, a.N) ? diff_fp64(__ldg(a.X + (size_t)ij.x * a.n + l), __ldg(a.X + (size_t)ij.y * a.n + l)) : 0.0;
            }
            meet();
            if (direct) {
                if (warp <= k)
                    for (int q = 0; q < nq; ++q) {
                        const double *D = Ds + (size_t)q * a.n;
                        double v = 0.0;
#pragma unroll
                        for (int t = 0; t < kSliceN / 32; ++t)
                            if (lane + 32 * t < a.n) {
                                const double d = D[lane + 32 * t];
                                v = fma(warp < k ? ur[t] : d, d, v);
                            }
                        v = warp_sum(v);
                        if (lane == 0) entries[q][warp] = v;
                    }
            } else
            for (int t = warp; t < nq * (k + 1); t += kConsumerWarps) {
                const int q = t / (k + 1), c = t - q * (k + 1);
                const double e = fp64_entry<true>(Ds + (size_t)q * a.n, a.U64, a.n, k, c, lane);
                if (lane == 0) entries[q][c] = e;
            }
            meet();
            if (warp < nq) {
                const int2 ij = packed_pair(queue[warp]);
                constexpr int KS = K <= 8 ? K : K <= 12 ? 12 : K <= 16 ? 16 : K <= 24 ? 24 : 32;
                double zz, d2;
                fp64_combine<KS>(entries[warp], a.n, k, lane, zz, d2);
                if (!(d2 == 0.0 || d2 < a.eps2)) {
                    const double q = zz / d2;
                    if (better_q(q, ij.x, ij.y, best.r, best.i, best.j)) best = Partial{q, ij.x, ij.y};
                }
            }
            if (tid == 0) atomicAdd((unsigned int *)&a.st->cnt2, (unsigned int)nq);
        }
        if (lane == 0) pbest[warp] = best;
    }
    __syncwarp();
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == kConsumerWarps + 1) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tbase, kTmemCols);
    }
    if (EXPL && tid == 0) {
        Partial b = pbest[0];
        for (int w2 = 1; w2 < kConsumerWarps; ++w2)
            if (better_q(pbest[w2].r, pbest[w2].i, pbest[w2].j, b.r, b.i, b.j)) b = pbest[w2];
        a.partials[blockIdx.x] = b;
    }
}

// ------------------------------------------- explicit-difference recheck ---

struct ExplArgs {
    const float *X;
    int N, n;
    const float *U32;  // n x KP
    const float *U32lo;  // n x KP, fl(U64 - U32) (extended-precision variant)
    int k, KP;
    const int2 *cand1;
    unsigned int cap1;
    const int2 *near;
    int n_near;
    Cert cert;
    ProbState *st;
    int2 *cand2;
    long long cap2;
    int pdl;
    int pack;          // extended-precision kernel: write cand2 as packed (i, j, ratio) entries
};

constexpr int EPW = 4;  // entries per warp per round

// Re-evaluates the pass's candidates and the near pairs from explicit FP32
// differences (error model of plain.cu), one warp per pair, and emits the
// pairs that can still be the argmin for the FP64 tier.  A warp handles EPW
// pairs per round with their loads interleaved, so a round costs one memory
// latency; the EPW*(K+1) warp sums are reduced together.  K is the compute
// width (k, or k rounded up; U32's pad columns are zero).
template <int K>
__global__ void __launch_bounds__(256) explicit_recheck_kernel(ExplArgs a)
{
    constexpr int KU = (K + 3) / 4 * 4;
    __shared__ float red[32];
    __shared__ int scan[33];
    __shared__ int base_sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // The near list is fixed and the basis and bounds are the previous
    // iteration's (complete once this kernel runs): it is evaluated while the
    // pass may still be running.  The pass's candidates follow its end.
    // With programmatic launch the lists are two segments (the near list
    // first, while the pass may still run; then, after the wait, the pass's
    // candidates); otherwise one segment covering both.
    const float seed = load_pos_float(&a.st->seed_ub);
    for (int seg = 0; seg < (a.pdl ? 2 : 1); ++seg) {
    long long nn = a.n_near, total = a.n_near, lim = a.n_near;
    if (seg == 1 || !a.pdl) {
        grid_dep_wait();
        grid_dep_launch();
        unsigned int c1 = *(volatile const unsigned int *)&a.st->cnt1;
        if (c1 > a.cap1) c1 = a.cap1;
        nn = a.pdl ? 0 : a.n_near;
        total = nn + c1;
        lim = nn + a.cap1;  // bound of the lists' storage
    }
    // A round's pairs are read up to the lists' storage bound before the
    // count is needed (entries past the count are read but not used), so the
    // count's load and the pairs' loads overlap.
    for (long long base = (long long)blockIdx.x * 8 * EPW; base < lim;
         base += (long long)gridDim.x * 8 * EPW) {
        int2 pr[EPW];
        bool valid[EPW];
#pragma unroll
        for (int e = 0; e < EPW; ++e) {
            const long long idx = base + warp * EPW + e;
            pr[e] = idx < lim ? (idx < nn ? __ldcg(a.near + idx) : __ldcg(a.cand1 + (idx - nn))) : make_int2(0, 0);
        }
        if (base >= total) break;  // uniform over the block
#pragma unroll
        for (int e = 0; e < EPW; ++e) {
            valid[e] = base + warp * EPW + e < total && SAP_PAIR_OK(a.st, pr[e], a.N);
            if (!valid[e]) pr[e] = make_int2(0, 0);
        }
        // any earlier value of the running bound is a valid (looser) bound:
        // read it now, so its latency overlaps the loads below
        const float ub2 = load_pos_float(&a.st->run_ub2);
        float acc[EPW * (K + 1)];
#pragma unroll
        for (int q = 0; q < EPW * (K + 1); ++q) acc[q] = 0.f;
#pragma unroll 2
        for (int l = lane; l < a.n; l += 32) {
            float u[KU];
#pragma unroll
            for (int c = 0; c < KU; c += 4) {
                const float4 t = __ldcg(reinterpret_cast<const float4 *>(a.U32 + (size_t)l * a.KP + c));
                u[c] = t.x; u[c + 1] = t.y; u[c + 2] = t.z; u[c + 3] = t.w;
            }
#pragma unroll
            for (int e = 0; e < EPW; ++e) {
                const float D = a.X[(size_t)pr[e].x * a.n + l] - a.X[(size_t)pr[e].y * a.n + l];
                acc[e * (K + 1) + K] = fmaf(D, D, acc[e * (K + 1) + K]);
#pragma unroll
                for (int c = 0; c < K; ++c) acc[e * (K + 1) + c] = fmaf(u[c], D, acc[e * (K + 1) + c]);
            }
        }
        // lane e < EPW finishes entry e: |D|^2 in z[K], U^T D in z[0..K-1]
        float z[K + 1];
        constexpr int M = EPW * (K + 1);
        if constexpr (M <= 32) {
            // reduce-scatter (M - 1 + a few shuffles instead of 5 M), then
            // each finishing lane gathers its entry's K + 1 totals
            constexpr int S = M <= 8 ? 8 : M <= 16 ? 16 : 32;
            constexpr int dup = 32 / S;  // lanes holding the same total
            float r[S];
#pragma unroll
            for (int q = 0; q < S; ++q) r[q] = q < M ? acc[q < M ? q : 0] : 0.f;
            const float t = warp_reduce_scatter<S>(r, lane);
            const int e = lane < EPW ? lane : 0;
#pragma unroll
            for (int c = 0; c <= K; ++c) z[c] = __shfl_sync(0xffffffffu, t, (e * (K + 1) + c) * dup);
        } else {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q < M; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
#pragma unroll
            for (int c = 0; c <= K; ++c) z[c] = acc[c];
#pragma unroll
            for (int e = 1; e < EPW; ++e)
                if (lane == e)
#pragma unroll
                    for (int c = 0; c <= K; ++c) z[c] = acc[e * (K + 1) + c];
        }
        int2 mypr = pr[0];
        bool myvalid = valid[0];
#pragma unroll
        for (int e = 1; e < EPW; ++e)
            if (lane == e) { mypr = pr[e]; myvalid = valid[e]; }
        const float dd = z[K];
        float zz = 0.f;
#pragma unroll
        for (int c = 0; c < K; ++c) zz = fmaf(z[c], z[c], zz);
        const int code = (lane >= EPW || !myvalid) ? 0 : (dd < 1e-30f ? 2 : 1);  // 2: too short for FP32
        const float rr = code == 1 ? sqrtf(zz / dd) : INFINITY;
        const float bmin = block_min(rr, red);
        float U = fminf(seed, ub2);
        if (bmin < INFINITY) {
            const float ub = cert_upper(bmin, a.cert);
            if (threadIdx.x == 0) atomic_min_pos_float(&a.st->run_ub2, ub);
            U = fminf(U, ub);
        }
        const float th = cert_emit_threshold(U, a.cert);
        const int cnt = (code == 2 || (code == 1 && rr <= th)) ? 1 : 0;
        int tot;
        const int off = block_exclusive_scan(cnt, scan, &tot);
        if (tot == 0) continue;
        if (threadIdx.x == 0) base_sh = (int)atomicAdd((unsigned int *)&a.st->cnt2, (unsigned int)tot);
        __syncthreads();
        if (cnt) {
            const long long pos = (long long)(unsigned int)base_sh + off;
            if (pos < a.cap2) a.cand2[pos] = mypr;
            else atomicOr(&a.st->status, ST_OVERFLOW);
        }
        __syncthreads();
    }
    }
}

// ---- extended-precision explicit recheck (large n; helpers in sap_internal.cuh)

// The same tier for large n, where the FP32 dot products' certified error
// (gamma_{n+3}) would pass too many pairs on: D = fl(x_i - x_j) in FP32, then
// |D|^2 and U^T D accumulated as hi + lo FP32 pairs with error-free products
// against the hi + lo FP32 basis.  Since U is orthonormal, the rounding of D
// moves U^T D by at most 2^-24 d and d by 2^-24 d, so |r~ - r| <= 2^-24 +
// 2 * 2^-24 r plus the final FP32 roundings (cert_explicit_df).  One warp per
// pair, K + 1 extended accumulators per lane.
template <int K>
__global__ void __launch_bounds__(256) explicit_df_kernel(ExplArgs a)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // pairs per warp and round: as many as the reduce-scatter holds
    constexpr int E = (K + 1) <= 8 ? 4 : (K + 1) <= 16 ? 2 : 1;
    // near list first (while the pass may still run), then the pass's candidates
    const float seed = load_pos_float(&a.st->seed_ub);
    for (int seg = 0; seg < (a.pdl ? 2 : 1); ++seg) {
    long long nn = a.n_near, total = a.n_near;
    if (seg == 1 || !a.pdl) {
        grid_dep_wait();
        grid_dep_launch();
        unsigned int c1 = *(volatile const unsigned int *)&a.st->cnt1;
        if (c1 > a.cap1) c1 = a.cap1;
        nn = a.pdl ? 0 : a.n_near;
        total = nn + c1;
    }
    for (long long base = ((long long)blockIdx.x * 8 + warp) * E; base < total; base += (long long)gridDim.x * 8 * E) {
        int2 pr[E];
        bool valid[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const long long idx = base + e;
            valid[e] = idx < total;
            pr[e] = valid[e] ? (idx < nn ? __ldcg(a.near + idx) : __ldcg(a.cand1 + (idx - nn))) : make_int2(0, 0);
            if (valid[e] && !SAP_PAIR_OK(a.st, pr[e], a.N)) {
                valid[e] = false;
                pr[e] = make_int2(0, 0);
            }
        }
        // any earlier value of the running bound is a valid (looser) bound
        const float ub2 = load_pos_float(&a.st->run_ub2);
        float rr;
        int code;
        if constexpr ((K + 1) * E <= 32) {
            df_eval<K, E>(a.X, a.n, a.U32, a.U32lo, a.KP, pr, valid, lane, rr, code);
        } else {
            // k = 32: K + 1 sums per pair, one pair per warp, butterfly sums
            float zh[K + 1], zl[K + 1];
#pragma unroll
            for (int q = 0; q <= K; ++q) zh[q] = zl[q] = 0.f;
            if (valid[0]) {
#pragma unroll 2
                for (int l = lane; l < a.n; l += 32) {
                    const float D = a.X[(size_t)pr[0].x * a.n + l] - a.X[(size_t)pr[0].y * a.n + l];
                    xs_fma(zh[K], zl[K], D, D, 0.f);
                    const float *uh = a.U32 + (size_t)l * a.KP, *ul = a.U32lo + (size_t)l * a.KP;
#pragma unroll
                    for (int c = 0; c < K; ++c) xs_fma(zh[c], zl[c], D, __ldcg(uh + c), __ldcg(ul + c));
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q <= K; ++q) {
                    const float h2 = __shfl_xor_sync(0xffffffffu, zh[q], o);
                    const float l2 = __shfl_xor_sync(0xffffffffu, zl[q], o);
                    float s, e;
                    xs_two_sum(zh[q], h2, s, e);
                    zh[q] = s;
                    zl[q] = __fadd_rn(zl[q], __fadd_rn(l2, e));
                }
            const float dd = zh[K] + zl[K];
            float zz = 0.f;
#pragma unroll
            for (int c = 0; c < K; ++c) {
                const float z = zh[c] + zl[c];
                zz = fmaf(z, z, zz);
            }
            code = (lane != 0 || !valid[0]) ? 0 : (dd < 1e-30f ? 2 : 1);  // 2: too short for FP32
            rr = code == 1 ? sqrtf(zz / dd) : INFINITY;
        }
        const float wmin = warp_min(rr);
        float U = fminf(seed, ub2);
        if (wmin < INFINITY) {
            const float ub = cert_upper(wmin, a.cert);
            if (lane == 0 && ub < ub2) atomic_min_pos_float(&a.st->run_ub2, ub);
            U = fminf(U, ub);
        }
        const float th = cert_emit_threshold(U, a.cert);
        const bool emit = code == 2 || (code == 1 && rr <= th);
        const unsigned int m = __ballot_sync(0xffffffffu, emit);
        if (!m) continue;
        unsigned int b0 = 0;
        if (lane == 0) b0 = atomicAdd((unsigned int *)&a.st->cnt2, (unsigned int)__popc(m));
        b0 = __shfl_sync(0xffffffffu, b0, 0);
        int2 mp = pr[0];
#pragma unroll
        for (int e = 1; e < E; ++e)
            if (lane == e) mp = pr[e];
        if (emit) {
            const long long pos = (long long)b0 + __popc(m & ((1u << lane) - 1u));
            if (pos < a.cap2) {
                if (a.pack) reinterpret_cast<unsigned long long *>(a.cand2)[pos] = pack_cand(mp.x, mp.y, rr, code == 2);
                else a.cand2[pos] = mp;
            } else {
                atomicOr(&a.st->status, ST_OVERFLOW);
            }
        }
    }
    }
}

template <int K>
cudaError_t launch_expl_k(const ExplArgs &x, bool df, int grid, cudaStream_t s)
{
    if (df) return launch_pdl(x.pdl != 0, explicit_df_kernel<K>, dim3(grid), dim3(256), 0, s, x);
    return launch_pdl(x.pdl != 0, explicit_recheck_kernel<K>, dim3(grid), dim3(256), 0, s, x);
}

cudaError_t launch_explicit(const ExplArgs &x, bool df, int grid, cudaStream_t s)
{
    switch (x.k) {
    case 1: return launch_expl_k<1>(x, df, grid, s);
    case 2: return launch_expl_k<2>(x, df, grid, s);
    case 3: return launch_expl_k<3>(x, df, grid, s);
    case 4: return launch_expl_k<4>(x, df, grid, s);
    case 5: return launch_expl_k<5>(x, df, grid, s);
    case 6: return launch_expl_k<6>(x, df, grid, s);
    case 7: return launch_expl_k<7>(x, df, grid, s);
    case 8: return launch_expl_k<8>(x, df, grid, s);
    default: break;
    }
    if (x.k <= 12) return launch_expl_k<12>(x, df, grid, s);
    if (x.k <= 16) return launch_expl_k<16>(x, df, grid, s);
    if (x.k <= 24) return launch_expl_k<24>(x, df, grid, s);
    return launch_expl_k<32>(x, df, grid, s);
}

// ------------------------------------------ the double-float refine tier ---
//
// Y is formed a second time per iteration in double-float arithmetic: every
// entry an unevaluated sum hi + lo of two FP32 numbers, from the exact FP32
// points (not centred: centring in FP32 would round the differences this
// tier exists to resolve) and the basis split as U32 + U32lo.  Each step is
// an error-free product x * uh (FMA residual), an error-free sum into hi, the
// small terms added to lo, and a renormalisation (|lo| <= ulp(hi)/2), so a
// step adds at most 9 * 2^-48 * S to the error, S = sum_l |x_l||u_l| <=
// ||x|| (u a unit vector); the split residual of u adds 2^-48 S and the five
// five lane merges 20 * 2^-48 S.  Hence |y~_c - y_c| <= eps_df ||x_i|| with
// eps_df = 1.25 (9n + 60) 2^-48 (about 4e-12 at n = 100).
//
// The refine tier evaluates every candidate of the pass and every near pair
// from these rows, one thread per pair, O(k) work: z_c = (yh_i - yh_j) +
// (yl_i - yl_j) (relative FP32 roundings only), r~ = |z| sqrt(w_ij) with the
// stored 1/d^2 (near pairs keep theirs in near_w).  Certified error
// |r~ - r| <= A_p + rho r, A_p = sqrt(k) (eps_df + 2^-46)(||x_i|| + ||x_j||)
// sqrt(w_ij): at least a thousand times below the pass's bound, and below the
// FP32 rounding of explicit differences x_i - x_j.  Emission as in every
// tier: r~_p <= U (1 + rho) + A_p against the running upper bound U.

double df_error_unit(int n)
{
    return 1.25 * (9.0 * n + 60.0) * std::ldexp(1.0, -48);
}

__device__ __forceinline__ void df_two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (hi, lo) += x * (uh + ul), then renormalised.  The _rn intrinsics keep the
// compiler from fusing the error-free steps into FMAs.
__device__ __forceinline__ void df_step(float &hi, float &lo, float x, float uh, float ul)
{
    const float p = __fmul_rn(x, uh);
    const float pe = fmaf(x, uh, -p);
    float s, e;
    df_two_sum(hi, p, s, e);
    const float l = __fadd_rn(lo, __fadd_rn(e, fmaf(x, ul, pe)));
    hi = __fadd_rn(s, l);
    lo = __fsub_rn(l, __fsub_rn(hi, s));
}
struct YdfArgs {
    const float *X;          // N x n row-major FP32
    int N, n;
    const float *U32, *U32lo;  // n x KP: hi and lo parts of the basis
    int KP;
    int Npad;
    float *Yh, *Yl;          // KY x Npad each, component-major; rows >= N zero
    int KY;
    // pair mode (st set, no more than pair_max pairs left by the pass)
    ProbState *st = nullptr;
    long long pair_max = -1;
    const int2 *cand1 = nullptr, *near_list = nullptr;
    Cert cert;               // of the extended-precision explicit evaluation
    unsigned long long *cand2 = nullptr;
    long long cap2 = 0;
};

// The pass left few pairs: they are evaluated one by one (pair mode) and the
// whole double-float Y is not needed.
__device__ __forceinline__ bool pair_mode(const ProbState *st, long long pair_max)
{
    const long long c = (long long)*(volatile const unsigned int *)&st->cnt1 + *(volatile const unsigned int *)&st->cntn;
    return c <= pair_max;
}

__device__ __forceinline__ void df_merge_norm(float &hi, float &lo, float h2, float l2)
{
    float s, e;
    df_two_sum(hi, h2, s, e);
    const float l = __fadd_rn(lo, __fadd_rn(l2, e));
    hi = __fadd_rn(s, l);
    lo = __fsub_rn(l, __fsub_rn(hi, s));
}

// Pair mode: a Y row costs n k error-free steps whether or not a candidate
// needs it, and N rows for a basis are 4 GFLOP of FP32 steps at N = n = 4096, k =
// 20 (0.3-0.5 ms beside the other bases' kernels); a pair costs n (k + 1).
// With fewer pairs than points a warp takes a pair instead, its differences
// in place of the row's coordinates and |D|^2 as one more component, and emits
// what the bound does not exclude for the FP64 tier (the error model of the
// extended-precision explicit tier).
//
// A block of 16 warps computes 32 rows at a time, two per warp; the lanes of
// a warp split the coordinates (l = lane, lane + 32, ...), and their partial
// sums are merged by a 5-level shuffle tree at the end (within the error
// allowance above).  The basis goes through shared memory in chunks of CH
// coordinates, component-major (lanes read consecutive words), each chunk
// serving all 32 rows.  K = compute width (U32's pad columns are zero).
constexpr int kYdfWarps = 16;
constexpr int kYdfRpw = 2;

template <int K>
struct YdfShape {
    static constexpr int CH = K <= 8 ? 256 : 128;
};

template <int K>
__global__ void __launch_bounds__(kYdfWarps * 32) ydf_warp_kernel(YdfArgs a)
{
    constexpr int CH = YdfShape<K>::CH;
    __shared__ float us[2 * K][CH];  // [c][l] hi, [K + c][l] lo
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nchunks = (a.n + CH - 1) / CH;
    if (a.st && pair_mode(a.st, a.pair_max)) {
        const int cn = *(volatile const int *)&a.st->cntn, total = *(volatile const int *)&a.st->cnt1 + cn;
        const float seed = load_pos_float(&a.st->seed_ub);
        for (int pbase = blockIdx.x * kYdfWarps; pbase < total; pbase += gridDim.x * kYdfWarps) {
            const int p = pbase + warp;
            int2 pr = make_int2(0, 0);
            bool valid = p < total;
            if (valid) {
                pr = p < cn ? __ldcg(a.near_list + p) : __ldcg(a.cand1 + (p - cn));
                valid = SAP_PAIR_OK(a.st, pr, a.N);
                if (!valid) pr = make_int2(0, 0);
            }
            const float *xi = a.X + (size_t)pr.x * a.n, *xj = a.X + (size_t)pr.y * a.n;
            float hi[K + 1], lo[K + 1];
#pragma unroll
            for (int c = 0; c <= K; ++c) hi[c] = lo[c] = 0.f;
            for (int ch = 0; ch < nchunks; ++ch) {
                const int c0 = ch * CH, nc = min(CH, a.n - c0);
                __syncthreads();
                for (int idx = threadIdx.x; idx < K * CH; idx += kYdfWarps * 32) {
                    const int c = idx / CH, l = idx % CH;
                    const bool in = l < nc;
                    us[c][l] = in ? a.U32[(size_t)(c0 + l) * a.KP + c] : 0.f;
                    us[K + c][l] = in ? a.U32lo[(size_t)(c0 + l) * a.KP + c] : 0.f;
                }
                __syncthreads();
                if (valid)
#pragma unroll 2
                    for (int l = lane; l < nc; l += 32) {
                        const float D = xi[c0 + l] - xj[c0 + l];
#pragma unroll
                        for (int c = 0; c < K; ++c) df_step(hi[c], lo[c], D, us[c][l], us[K + c][l]);
                        df_step(hi[K], lo[K], D, D, 0.f);
                    }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c <= K; ++c) {
                    const float h2 = __shfl_xor_sync(0xffffffffu, hi[c], o);
                    const float l2 = __shfl_xor_sync(0xffffffffu, lo[c], o);
                    df_merge_norm(hi[c], lo[c], h2, l2);
                }
            if (lane == 0 && valid) {
                const float dd = hi[K];
                float zz = 0.f;
#pragma unroll
                for (int c = 0; c < K; ++c) zz = fmaf(hi[c], hi[c], zz);
                float lb = 0.f;  // too short for FP32: the FP64 tier decides
                float U = fminf(seed, fminf(load_pos_float(&a.st->run_ub1), load_pos_float(&a.st->run_ub2)));
                if (!(dd < 1e-30f)) {
                    const float rr = sqrtf(zz / dd), ub = cert_upper(rr, a.cert);
                    if (ub < U) atomic_min_pos_float(&a.st->run_ub2, ub);
                    U = fminf(U, ub);
                    lb = fmaxf((rr - a.cert.A) / (1.0f + a.cert.rho) * 0.999998f, 0.f);
                }
                if (lb <= U * 1.000001f) {
                    const unsigned int at = atomicAdd((unsigned int *)&a.st->cnt2, 1u);
                    if ((long long)at < a.cap2) a.cand2[at] = pack_cand(pr.x, pr.y, lb, lb == 0.f);
                    else atomicOr(&a.st->status, ST_OVERFLOW);
                }
            }
        }
        return;
    }
    for (int rbase = blockIdx.x * (kYdfWarps * kYdfRpw); rbase < a.Npad;
         rbase += gridDim.x * (kYdfWarps * kYdfRpw)) {
        float hi[kYdfRpw][K], lo[kYdfRpw][K];
#pragma unroll
        for (int q = 0; q < kYdfRpw; ++q)
#pragma unroll
            for (int c = 0; c < K; ++c) hi[q][c] = lo[q][c] = 0.f;
        for (int ch = 0; ch < nchunks; ++ch) {
            const int c0 = ch * CH, nc = min(CH, a.n - c0);
            if (nchunks > 1 || rbase == blockIdx.x * (kYdfWarps * kYdfRpw)) {
                __syncthreads();
                for (int idx = threadIdx.x; idx < K * CH; idx += kYdfWarps * 32) {
                    const int c = idx / CH, l = idx % CH;
                    const bool in = l < nc;
                    us[c][l] = in ? a.U32[(size_t)(c0 + l) * a.KP + c] : 0.f;
                    us[K + c][l] = in ? a.U32lo[(size_t)(c0 + l) * a.KP + c] : 0.f;
                }
                __syncthreads();
            }
#pragma unroll
            for (int q = 0; q < kYdfRpw; ++q) {
                const int row = rbase + warp * kYdfRpw + q;
                if (row >= a.N) continue;
                const float *xr = a.X + (size_t)row * a.n + c0;
#pragma unroll 2
                for (int l = lane; l < nc; l += 32) {
                    const float x = xr[l];
#pragma unroll
                    for (int c = 0; c < K; ++c) df_step(hi[q][c], lo[q][c], x, us[c][l], us[K + c][l]);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kYdfRpw; ++q) {
            const int row = rbase + warp * kYdfRpw + q;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < K; ++c) {
                    const float h2 = __shfl_xor_sync(0xffffffffu, hi[q][c], o);
                    const float l2 = __shfl_xor_sync(0xffffffffu, lo[q][c], o);
                    df_merge_norm(hi[q][c], lo[q][c], h2, l2);
                }
            if (row < a.Npad)
#pragma unroll
                for (int c = 0; c < K; ++c)
                    if (lane == c % 32 && c < a.KY) {
                        a.Yh[(size_t)c * a.Npad + row] = hi[q][c];
                        a.Yl[(size_t)c * a.Npad + row] = lo[q][c];
                    }
        }
    }
}

struct RefineArgs {
    const float *Yh, *Yl;    // double-float Y, KY x Npad each
    int Npad;
    const float *w;          // stored 1/d^2, tile-major upper triangle
    int nb;                  // point blocks per side (Npad / 128)
    long long tile0;         // global index of the first stored tile
    long long nwt;           // stored tiles (index checks of the debug build)
    const float *xn;         // ||x_i||, rounded up
    float beta;              // sqrt(k) (eps_df + 2^-46), rounded up
    const int2 *cand1;
    unsigned int cap1;
    const int2 *near;
    const float *near_w;     // 1/d^2 of the near pairs (+inf: too short for FP32)
    int n_near;
    Cert cert;               // rho (A unused: each pair has its own bound)
    ProbState *st;
    unsigned long long *cand2;  // packed (i, j, lower bound of the ratio)
    long long cap2;
    int pdl;
    long long pair_max;      // the double-float kernel took the pairs itself up to this many
};

// One thread per pair; K = compute width (Y's pad components are zero).
// Warps aggregate their bound and their emissions (one atomic each).
template <int K>
__global__ void __launch_bounds__(256) refine_kernel(RefineArgs a)
{
    const int lane = threadIdx.x & 31;
    const float rho = a.cert.rho;
    grid_dep_wait();
    grid_dep_launch();
    if (pair_mode(a.st, a.pair_max)) return;
    const float seed = load_pos_float(&a.st->seed_ub);
    {
        long long nn = a.n_near, total = a.n_near;
        {
            unsigned int c1 = *(volatile const unsigned int *)&a.st->cnt1;
            if (c1 > a.cap1) c1 = a.cap1;
            total = nn + c1;
        }
        const long long stride = (long long)gridDim.x * blockDim.x;
        // rounds are warp-uniform: every lane of a warp runs the same count
        for (long long base = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < total;
             base += stride) {
            const long long idx = base + lane;
            const float Uround = fminf(seed, load_pos_float(&a.st->run_ub2));  // issued early
            int code = 0;  // 0 none, 1 evaluated, 2 too short for FP32 (always emitted)
            int2 pr = make_int2(0, 0);
            float r = INFINITY, bnd = 0.f;
            if (idx < total) {
                float wv = INFINITY;
                bool ok;
                if (idx < nn) {
                    pr = __ldcg(a.near + idx);
                    ok = SAP_BOUNDS_OK(a.st, pr.x >= 0 && pr.x < pr.y && pr.y < a.Npad);
                    wv = __ldcg(a.near_w + idx);
                } else {
                    pr = __ldcg(a.cand1 + (idx - nn));
                    const int I = pr.x >> 7, J = pr.y >> 7;
                    const long long t = (long long)I * a.nb - (long long)I * (I - 1) / 2 + (J - I) - a.tile0;
                    ok = SAP_BOUNDS_OK(a.st, pr.x >= 0 && pr.x < pr.y && pr.y < a.Npad && t >= 0 && t < a.nwt);
                    if (ok) wv = __ldg(a.w + t * (T * T) + (pr.x & (T - 1)) * T + (pr.y & (T - 1)));
                }
                if (!ok) {
                    pr = make_int2(0, 0);  // skipped (code 0)
                } else if (!(wv < INFINITY)) {
                    code = 2;
                } else {
                    float zz = 0.f;
#pragma unroll
                    for (int c = 0; c < K; ++c) {
                        const size_t oi = (size_t)c * a.Npad + pr.x, oj = (size_t)c * a.Npad + pr.y;
                        const float z = __fadd_rn(__fsub_rn(__ldcg(a.Yh + oi), __ldcg(a.Yh + oj)),
                                                  __fsub_rn(__ldcg(a.Yl + oi), __ldcg(a.Yl + oj)));
                        zz = fmaf(z, z, zz);
                    }
                    const float sw = sqrtf(wv);
                    r = sqrtf(zz * wv);
                    bnd = a.beta * (__ldg(a.xn + pr.x) + __ldg(a.xn + pr.y)) * sw * 1.000002f;
                    code = 1;
                }
            }
            // the warp's best upper bound tightens the running bound
            const float ub = code == 1 ? (r + bnd) / (1.0f - rho) * 1.000001f : INFINITY;
            const float wub = warp_min(ub);
            float U = Uround;
            if (wub < U) {
                if (lane == 0) atomic_min_pos_float(&a.st->run_ub2, wub);
                U = wub;
            }
            const bool emit = code == 2 || (code == 1 && r <= (U * (1.0f + rho) + bnd) * 1.000001f);
            const unsigned m = __ballot_sync(0xffffffffu, emit);
            if (m) {
                unsigned int b = 0;
                if (lane == 0) b = atomicAdd((unsigned int *)&a.st->cnt2, (unsigned int)__popc(m));
                b = __shfl_sync(0xffffffffu, b, 0);
                if (emit) {
                    const long long pos = (long long)b + __popc(m & ((1u << lane) - 1u));
                    // with a lower bound on its ratio, against which the FP64
                    // recheck filters once the bound is final (rounded down)
                    const float lb = code == 2 ? 0.f : fmaxf((r - bnd) / (1.0f + rho) * 0.999998f, 0.f);
                    if (pos < a.cap2) a.cand2[pos] = pack_cand(pr.x, pr.y, lb, code == 2);
                    else atomicOr(&a.st->status, ST_OVERFLOW);
                }
            }
        }
    }
}

template <int K>
cudaError_t launch_ydf_refine_k(const YdfArgs &y, const RefineArgs &x, int ygrid, int rgrid, bool ydf,
                                cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    if (ydf) {
        const int need = (y.Npad + kYdfWarps * kYdfRpw - 1) / (kYdfWarps * kYdfRpw);
        ydf_warp_kernel<K><<<std::min(need, ygrid), kYdfWarps * 32, 0, s>>>(y);
        e = cudaGetLastError();
    } else {
        e = launch_pdl(x.pdl != 0, refine_kernel<K>, dim3(rgrid), dim3(256), 0, s, x);
    }
    return e;
}

// The double-float product (ydf = true) or the refine tier, for width k.
cudaError_t launch_ydf_refine(const YdfArgs &y, const RefineArgs &x, int k, int ygrid, int rgrid, bool ydf,
                              cudaStream_t s)
{
    switch (k) {
    case 1: return launch_ydf_refine_k<1>(y, x, ygrid, rgrid, ydf, s);
    case 2: return launch_ydf_refine_k<2>(y, x, ygrid, rgrid, ydf, s);
    case 3: return launch_ydf_refine_k<3>(y, x, ygrid, rgrid, ydf, s);
    case 4: return launch_ydf_refine_k<4>(y, x, ygrid, rgrid, ydf, s);
    case 5: return launch_ydf_refine_k<5>(y, x, ygrid, rgrid, ydf, s);
    case 6: return launch_ydf_refine_k<6>(y, x, ygrid, rgrid, ydf, s);
    case 7: return launch_ydf_refine_k<7>(y, x, ygrid, rgrid, ydf, s);
    case 8: return launch_ydf_refine_k<8>(y, x, ygrid, rgrid, ydf, s);
    default: break;
    }
    if (k <= 12) return launch_ydf_refine_k<12>(y, x, ygrid, rgrid, ydf, s);
    if (k <= 16) return launch_ydf_refine_k<16>(y, x, ygrid, rgrid, ydf, s);
    if (k <= 24) return launch_ydf_refine_k<24>(y, x, ygrid, rgrid, ydf, s);
    return launch_ydf_refine_k<32>(y, x, ygrid, rgrid, ydf, s);
}

// -------------------------------------------------------------- host side --

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

// 2-D map of a row-major [outer x inner] 16-bit matrix, box [box_outer x 64]
// with 128-byte swizzling (the K-major operand layout of the product).
bool make_map(CUtensorMap *m, void *base, bool bf16, uint64_t inner, uint64_t outer, uint32_t box_outer)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {inner * 2};
    cuuint32_t box[2] = {64, box_outer};
    cuuint32_t es[2] = {1, 1};
    return fn(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, dims,
              strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// block-major Y ([Npad/128][KY][128]) -> N x k row-major
__global__ void transpose_y_kernel(const float *Yb, int KY, int N, int k, float *out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N * k) return;
    const int i = e / k, c = e % k;
    out[e] = Yb[(size_t)(i >> 7) * KY * 128 + (size_t)c * 128 + (i & 127)];
}

template <typename T_>
void dfree(T_ *&p)
{
    if (p) cudaFree(p);
    p = nullptr;
}

#define RCK(call)                                                                            \
    do {                                                                                     \
        cudaError_t e_ = (call);                                                             \
        if (e_ != cudaSuccess)                                                               \
            return handle_fail(h, e_ == cudaErrorMemoryAllocation ? SAP_E_OOM : SAP_E_CUDA,  \
                               cudaGetErrorString(e_));                                      \
    } while (0)

// Bound on |y~_c - y_c| per unit ||fl(x - mean)|| (see gemm_tc.cu):
// centring and epilogue roundings, the split residuals and dropped low
// product, the FP32 accumulation chain of the high product within a K slice
// (ceil(NP/(16 ksplit)) MMAs, plus slack for the in-instruction adder
// tree), each accumulation step bounded by 2^-23 (truncation) of twice the
// running magnitude, and the FP32 sum of the slices.  Times 1.25 for margin.
double y_error_unit(int NP, bool bf16, int ksplit)
{
    const double u = std::ldexp(1.0, -24);
    const double split = bf16 ? 3.0 * std::ldexp(1.0, -16) : 3.0 * std::ldexp(1.0, -22);
    const double acc = (std::ceil(NP / (16.0 * ksplit)) + 4.0) * 2.0 * std::ldexp(1.0, -23);
    const double slices = (ksplit - 1) * 2.0 * u;  // FP32 sum of the K slices
    return (3.0 * u + split + acc + slices) * 1.25;
}

// K slices of the product: each slice at least 8 blocks of 64, at most 8
// slices (shorter FP32 accumulation chains for large n).
int pick_ksplit(int nkb) { return std::max(1, std::min(8, nkb / 8)); }

Cert cert_pass(int n, int k, double b_cap)
{
    const double u = std::ldexp(1.0, -24);
    auto g = [&](double m) { return m * u / (1.0 - m * u); };
    Cert c;
    c.A = (float)(b_cap * 1.002);  // >= every stored pair's own bound (FP32 rounding)
    // 2^-9: the BF16 rounding of w = 1/d^2 (halved by the square root); the
    // rest as for explicit differences
    c.rho = (float)((std::ldexp(1.0, -9) + g(n + 2) + g(k) + 8 * u) * 1.05);
    return c;
}

// Relative error of the pass's ratios with the FP32 w in place of the BF16 one.
float cert_pass32(int n, int k)
{
    const double u = std::ldexp(1.0, -24);
    auto g = [&](double m) { return m * u / (1.0 - m * u); };
    return (float)((g(n + 2) + g(k) + 8 * u) * 1.05);
}

// Explicit tier in extended precision for large n (the FP32 tier's
// gamma_{n+3} bound grows with n).
bool explicit_uses_df(int n) { return n > 256; }

Cert cert_explicit(int n, int k)
{
    const double u = std::ldexp(1.0, -24);
    auto g = [&](double m) { return m * u / (1.0 - m * u); };
    Cert c;
    c.A = (float)(std::sqrt((double)k) * g(n + 3) * 1.05);
    c.rho = (float)((g(n + 2) + g(k) + 3 * u) * 1.05);
    return c;
}

// Refine tier: relative errors only besides each pair's own bound (the
// rounding of the stored length, the FP32 differences, squares and sum of
// the k components, the product with w and the square root).
Cert cert_refine(int n, int k)
{
    const double u = std::ldexp(1.0, -24);
    auto g = [&](double m) { return m * u / (1.0 - m * u); };
    Cert c;
    c.A = 0.f;
    c.rho = (float)((g(n + 2) + g(k + 2) + 8 * u) * 1.05);
    return c;
}

sap_status classify(sap_handle h, int k)
{
    RestrState &r = restr_state(h);
    r.b_cap = handle_tune(h).b_cap;
    cudaStream_t s = handle_stream(h);
    RCK(cudaMemsetAsync(r.counters, 0, 8 * sizeof(unsigned int), s));
    WPrepArgs a;
    a.X = handle_x32(h);
    a.N = (int)handle_n_points(h);
    a.n = handle_n_dim(h);
    a.nu = r.nu;
    a.wtiles = r.wtiles;
    a.w = r.w;
    a.wb = reinterpret_cast<__nv_bfloat16 *>(r.wb);
    a.wb_scale = 1.0f / (r.yscale * r.yscale);
    a.eps2_lo = handle_eps2_lo(h);
    a.eps2_hi = handle_eps2_hi(h);
    a.eps2 = handle_eps2(h);
    a.beta_coef = (float)(std::sqrt((double)k) * r.y_eps * 1.02);
    a.b_cap = (float)r.b_cap;
    a.near = r.near;
    a.near_w = r.near_w;
    a.near_cap = r.near_cap;
    a.counters = r.counters;
    wprep_kernel<<<r.nwtiles, 256, 0, s>>>(a);
    RCK(cudaGetLastError());
    unsigned int cnt[8];
    RCK(cudaMemcpyAsync(cnt, r.counters, sizeof(cnt), cudaMemcpyDeviceToHost, s));
    RCK(cudaStreamSynchronize(s));
    if (cnt[2]) return handle_fail(h, SAP_E_UNSUPPORTED, "near-pair list overflow; raise the pass bound");
    r.n_near = (int)cnt[0];
    unsigned long long ex;
    std::memcpy(&ex, &cnt[4], sizeof(ex));
    r.n_excluded = (long long)ex;
    r.k_cls = k;
    return SAP_OK;
}

// The FP32 rows of Y are staged with a tile where that leaves three stages
// (the slow path then stays in shared memory); wider bases read them from L2.
bool pass_stages_y(int k) { return 3 * pass_stage_bytes(k, true) <= (uint32_t)kPassDynSmem; }

int pass_pick_stages(int k)
{
    int s = kPassStagesMax;
    while (s > 2 && s * pass_stage_bytes(k, pass_stages_y(k)) > (uint32_t)kPassDynSmem) --s;
    return s;
}

template <int K, bool EXPL>
cudaError_t launch_pass_k(const PassArgs &a, int grid, cudaStream_t s)
{
    const size_t shm = (size_t)a.stages * pass_stage_bytes(a.k, a.stage_y != 0);
    return launch_pdl(a.pdl != 0, restr_pass_kernel<K, EXPL>, dim3(grid), dim3(kPassThreads), shm, s, a);
}

template <int K, bool EXPL>
cudaError_t config_pass_k()
{
    return cudaFuncSetAttribute(restr_pass_kernel<K, EXPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPassDynSmem);
}

cudaError_t configure_pass_kernels()
{
    cudaError_t e = cudaSuccess;
    auto f = [&](cudaError_t x) { if (x != cudaSuccess) e = x; };
    f(config_pass_k<1, true>()); f(config_pass_k<2, true>()); f(config_pass_k<3, true>()); f(config_pass_k<4, true>());
    f(config_pass_k<5, true>()); f(config_pass_k<6, true>()); f(config_pass_k<7, true>()); f(config_pass_k<8, true>());
    f(config_pass_k<10, true>()); f(config_pass_k<12, true>()); f(config_pass_k<16, true>());
    f(config_pass_k<1, false>());
    return e;
}

// The form with the second tier inside exists for k <= 16.
cudaError_t launch_pass(const PassArgs &a, int grid, cudaStream_t s)
{
    if (!a.X) return launch_pass_k<1, false>(a, grid, s);
    switch (a.k) {
    case 1: return launch_pass_k<1, true>(a, grid, s);
    case 2: return launch_pass_k<2, true>(a, grid, s);
    case 3: return launch_pass_k<3, true>(a, grid, s);
    case 4: return launch_pass_k<4, true>(a, grid, s);
    case 5: return launch_pass_k<5, true>(a, grid, s);
    case 6: return launch_pass_k<6, true>(a, grid, s);
    case 7: return launch_pass_k<7, true>(a, grid, s);
    case 8: return launch_pass_k<8, true>(a, grid, s);
    default: break;
    }
    if (a.k <= 10) return launch_pass_k<10, true>(a, grid, s);
    if (a.k <= 12) return launch_pass_k<12, true>(a, grid, s);
    if (a.k <= 16) return launch_pass_k<16, true>(a, grid, s);
    return cudaErrorNotSupported;
}

// Errors of the filter's contraction per unit s_i + s_j (kappa) and absolute
// (kabs), in units of yscale, |y| <= 64: the two-term FP16 splits (dropped low
// product and residuals 3 2^-22, norms 2 2^-22, subnormal residuals 2^-25
// sqrt(k) relative and 2^-24 (sqrt(k) + 1) absolute), the FP32 sum of the
// norms, and per MMA step a truncation of 2^-23 of twice the running
// magnitude, itself at most 2 (s_i + s_j), plus slack for the adder tree.
void op_bounds(int k, float *kappa, float *kabs)
{
    const double u22 = std::ldexp(1.0, -22);
    const double kap = 5.0 * u22 + (k + 2) * std::ldexp(1.0, -24) + (op_ksteps(k) + 4) * std::ldexp(1.0, -21) +
                       std::sqrt((double)k) * std::ldexp(1.0, -25);
    *kappa = (float)(kap * 1.1);
    *kabs = (float)((std::sqrt((double)k) + 1.0) * std::ldexp(1.0, -24) * 1.1);
}

} // namespace

sap_status restructured_prepare(sap_handle h)
{
    RestrState &r = restr_state(h);
    cudaStream_t s = handle_stream(h);
    const int N = (int)handle_n_points(h), n = handle_n_dim(h);
    const bool bf16 = handle_split_bf16(h) != 0;
    const float *X = handle_x32(h);
    RCK(cudaStreamSynchronize(s));
    if (!r.center) {
        r.Npad = (N + T - 1) / T * T;
        r.NP = (n + 63) / 64 * 64;
        RCK(cudaMalloc(&r.center, n * sizeof(float)));
        RCK(cudaMalloc(&r.colpart, colmean_scratch(N, n) * sizeof(double)));
        RCK(cudaMalloc(&r.nu, r.Npad * sizeof(float)));
        RCK(cudaMalloc(&r.Xhi, (size_t)r.Npad * r.NP * 2));
        RCK(cudaMalloc(&r.Xlo, (size_t)r.Npad * r.NP * 2));
        RCK(cudaMalloc(&r.counters, 8 * sizeof(unsigned int)));
        const int nb = r.Npad / T;
        long long t0 = 0, t1 = -1;  // a shard stores the tiles [t0, t1) of the row-major order only
        handle_shard(h, &t0, &t1);
        std::vector<int2> t;
        long long g = 0;
        for (int I = 0; I < nb; ++I)
            for (int J = I; J < nb; ++J, ++g)
                if (g >= t0 && (t1 < 0 || g < t1)) t.push_back(make_int2(I, J));
        r.tile0 = t0;
        r.nwtiles = (int)t.size();
        RCK(cudaMalloc(&r.wtiles, t.size() * sizeof(int2)));
        RCK(cudaMemcpyAsync(r.wtiles, t.data(), t.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
        RCK(cudaStreamSynchronize(s));
        RCK(cudaMalloc(&r.w, (size_t)r.nwtiles * T * T * sizeof(float)));
        RCK(cudaMalloc(&r.wb, (size_t)r.nwtiles * T * T * sizeof(uint16_t)));
        const long long P = (long long)N * (N - 1) / 2;
        r.near_cap = (unsigned int)std::min<long long>(P + 64, 1ll << 24);
        RCK(cudaMalloc(&r.near, (size_t)r.near_cap * sizeof(int2)));
        RCK(cudaMalloc(&r.near_w, (size_t)r.near_cap * sizeof(float)));
        RCK(cudaMalloc(&r.xn, r.Npad * sizeof(float)));
        RCK(gemm_configure());
        RCK(update_cluster_configure());
        RCK(configure_pass_kernels());
    }
    const int sms = handle_sms(h);
    RCK(launch_colmean(X, N, n, r.colpart, r.center, s));
    RCK(cudaMemsetAsync(r.counters, 0, 8 * sizeof(unsigned int), s));
    absmax_kernel<<<4 * sms, 256, 0, s>>>(X, (size_t)N * n, n, r.center, r.counters);
    RCK(cudaGetLastError());
    unsigned int mbits = 0;
    RCK(cudaMemcpyAsync(&mbits, r.counters, sizeof(mbits), cudaMemcpyDeviceToHost, s));
    RCK(cudaStreamSynchronize(s));
    float mx;
    std::memcpy(&mx, &mbits, sizeof(mx));
    int e = 0;
    if (mx > 0.f) e = (int)std::ceil(std::log2((double)mx));
    r.xscale = (float)std::ldexp(1.0, -e);
    // |y| <= ||x - mean|| <= sqrt(n) 2^e (1 + eps_Y): scaled to at most 64
    r.yscale = (float)std::ldexp(1.0, 6 - e - (int)std::ceil(0.5 * std::log2((double)n) + 0.01));
    const float lo_mul = bf16 ? 256.f : 2048.f;
    if (bf16)
        split_kernel<__nv_bfloat16><<<4 * sms, 256, 0, s>>>(X, N, n, r.center, r.xscale, lo_mul,
                                                          (__nv_bfloat16 *)r.Xhi, (__nv_bfloat16 *)r.Xlo,
                                                          r.Npad, r.NP);
    else
        split_kernel<__half><<<4 * sms, 256, 0, s>>>(X, N, n, r.center, r.xscale, lo_mul, (__half *)r.Xhi,
                                                     (__half *)r.Xlo, r.Npad, r.NP);
    RCK(cudaGetLastError());
    rownorm_kernel<<<(r.Npad + 7) / 8, 256, 0, s>>>(X, N, n, r.center, r.nu, r.Npad);
    RCK(cudaGetLastError());
    xnorm_kernel<<<(r.Npad + 7) / 8, 256, 0, s>>>(X, N, n, r.xn, r.Npad);
    RCK(cudaGetLastError());
    r.ksplit = pick_ksplit(r.NP / 64);
    r.y_eps = y_error_unit(r.NP, bf16, r.ksplit);
    if (!make_map(&r.gemm.ta_hi, r.Xhi, bf16, r.NP, r.Npad, 128) ||
        !make_map(&r.gemm.ta_lo, r.Xlo, bf16, r.NP, r.Npad, 128))
        return handle_fail(h, SAP_E_CUDA, "cuTensorMapEncodeTiled failed for X");
    r.maps_x = true;
    if (r.Uhi) {
        if (!make_map(&r.gemm.tb_hi, r.Uhi, bf16, r.NP, r.KPG, r.KPG) ||
            !make_map(&r.gemm.tb_lo, r.Ulo, bf16, r.NP, r.KPG, r.KPG))
            return handle_fail(h, SAP_E_CUDA, "cuTensorMapEncodeTiled failed for U");
    }
    r.k_cls = 0;
    const int k = handle_k(h);
    if (k > 0) return classify(h, k);
    RCK(cudaStreamSynchronize(s));
    return SAP_OK;
}

sap_status restructured_basis_alloc(sap_handle h)
{
    RestrState &r = restr_state(h);
    const int k = handle_k(h);
    const bool bf16 = handle_split_bf16(h) != 0;
    cudaStream_t s = handle_stream(h);
    dfree(r.Uhi);
    dfree(r.Ulo);
    dfree(r.Y);
    dfree(r.ops);
    dfree(r.Ypart);
    r.KPG = (k + 15) / 16 * 16;
    r.KY = padded_stride(k);   // <= KPG; columns >= k are zero
    RCK(cudaMalloc(&r.Uhi, (size_t)r.KPG * r.NP * 2));
    RCK(cudaMalloc(&r.Ulo, (size_t)r.KPG * r.NP * 2));
    RCK(cudaMemsetAsync(r.Uhi, 0, (size_t)r.KPG * r.NP * 2, s));  // pad rows and columns stay zero
    RCK(cudaMemsetAsync(r.Ulo, 0, (size_t)r.KPG * r.NP * 2, s));
    RCK(cudaMalloc(&r.Y, (size_t)r.Npad * r.KY * sizeof(float)));
    RCK(cudaMemsetAsync(r.Y, 0, (size_t)r.Npad * r.KY * sizeof(float), s));
    const size_t op_bytes = (size_t)(r.Npad / T) * 2 * op_image_bytes(k);
    RCK(cudaMalloc(&r.ops, op_bytes));
    RCK(cudaMemsetAsync(r.ops, 0, op_bytes, s));  // pad halves stay zero
    dfree(r.near_list);
    RCK(cudaMalloc(&r.near_list, (size_t)handle_n_points(h) * sizeof(int2)));
    dfree(r.Ydh);
    dfree(r.Ydl);
    RCK(cudaMalloc(&r.Ydh, (size_t)r.Npad * r.KY * sizeof(float)));
    RCK(cudaMalloc(&r.Ydl, (size_t)r.Npad * r.KY * sizeof(float)));
    RCK(cudaMemsetAsync(r.Ydh, 0, (size_t)r.Npad * r.KY * sizeof(float), s));
    RCK(cudaMemsetAsync(r.Ydl, 0, (size_t)r.Npad * r.KY * sizeof(float), s));
    dfree(r.Ypart);
    if (r.ksplit > 1) RCK(cudaMalloc(&r.Ypart, (size_t)r.ksplit * r.Npad * r.KY * sizeof(float)));
    if (!make_map(&r.gemm.tb_hi, r.Uhi, bf16, r.NP, r.KPG, r.KPG) ||
        !make_map(&r.gemm.tb_lo, r.Ulo, bf16, r.NP, r.KPG, r.KPG))
        return handle_fail(h, SAP_E_CUDA, "cuTensorMapEncodeTiled failed for U");
    r.maps_u = true;
    return SAP_OK;
}

// The basis's operands were rewritten: the near list must fit its width.
sap_status restructured_basis_changed(sap_handle h)
{
    const int k = handle_k(h);
    if (restr_state(h).k_cls != k) return classify(h, k);
    return SAP_OK;
}

sap_status restructured_set_bound(sap_handle h, double b_cap)
{
    handle_tune(h).b_cap = b_cap;
    const int k = handle_k(h);
    if (k > 0) return classify(h, k);
    return SAP_OK;
}

GemmArgs product_args(sap_handle h, const RestrState &r)
{
    GemmArgs g = r.gemm;
    g.seed_st = nullptr;
    g.Npad = r.Npad;
    g.nkb = r.NP / 64;
    g.ab_bf16 = handle_split_bf16(h);
    g.lo_scale = g.ab_bf16 ? 1.0f / 256.f : 1.0f / 2048.f;
    g.out_scale = 1.0f / r.xscale;
    g.ksplit = r.ksplit;
    g.pdl = handle_tune(h).pdl;
    return g;
}

uint32_t restructured_op_groups(GemmArgs &g, const int *k, int count)
{
    uint32_t off = 0;
    int grp = 0;
    g.nbases = count;
    for (int q = 0; q < count; ++q) {
        float kappa, kabs;
        op_bounds(k[q], &kappa, &kabs);
        const int used = (k[q] + 3) / 4, all = padded_stride(k[q]) / 4;
        g.base_group[q] = grp;
        for (int c = 0; c < all; ++c)
            g.groups[grp++] = OpGroup{off, op_image_bytes(k[q]), c < used ? c : -1, c == used - 1, 1.0f - kappa, 0.5f * kabs};
        off += 2 * op_image_bytes(k[q]);
    }
    g.base_group[count] = grp;
    return off;
}

sap_status restructured_enqueue_product(sap_handle h, const CUtensorMap *mhi, const CUtensorMap *mlo, int KPG,
                                        float *Y, const OpsView &ops, int KY, float *Ypart, ProbState *st,
                                        cudaStream_t s, bool seeds)
{
    RestrState &r = restr_state(h);
    GemmArgs g = product_args(h, r);
    g.ops = ops.ops;
    g.ops_stride = restructured_op_groups(g, ops.k, ops.count);
    g.ops_scale = r.yscale;
    if (seeds) {
        g.seed_X = handle_x32(h);
        g.seed_U = handle_u32(h);
        g.seed_Ulo = handle_u32lo(h);
        g.seed_st = st;
        g.seed_N = (int)handle_n_points(h);
        g.seed_n = handle_n_dim(h);
        g.seed_k = handle_k(h);
        g.seed_KP = handle_kp(h);
    }
    g.tb_hi = *mhi;
    g.tb_lo = *mlo;
    g.Y = Y;
    g.KY = KY;
    g.KPG = KPG;
    g.stages = gemm_pick_stages(KPG, g.nkb, r.Npad / T * g.ksplit, handle_sms(h));
    g.st = st;
    g.Ypart = Ypart;
    cudaEvent_t ea, eb;
    handle_count_launch(h, 0, &ea, &eb);
    if (ea) cudaEventRecord(ea, s);
    RCK(launch_gemm_y(g, s));
    if (eb) cudaEventRecord(eb, s);
    handle_push_timing(h, 0, ea, eb);
    return SAP_OK;
}

// Does the pass of the double-float tier look at the near pairs itself, so that
// the pairs left can be evaluated one by one (pair mode)?  That takes the pass
// a gather of 2 k words per near pair, and pays only if it leaves at most N
// pairs.  us per iteration without and with it: 20 bases side by side over N =
// 4000 points, n = 2000, 4 000 near pairs 1754, 885; 159 000 1853, 1442; 319 000
// 1912, 1971; 799 000 2093, 3351; N = 1500 = n, 112 000 673, 538; 563 000 853,
// 1002; one basis (k = 6) over N = 3000, n = 300, 90 000 70, 68; 181 000 72, 78;
// 2 249 000 113, 261.  Hence at most 80 per point and a tenth of N n.
bool pairs_pay(long long N, int n, int k, long long n_near)
{
    return k <= 24 && n_near <= 80 * N && 10 * n_near <= N * n;
}

sap_status restructured_enqueue_basis(sap_handle h, const BasisView &b, cudaStream_t s)
{
    RestrState &r = restr_state(h);
    const int n = handle_n_dim(h);
    cudaEvent_t ea, eb;
    const int tier = restructured_tier_for(h, b.k);
    const bool pairs = tier == 1 && b.near_list && pairs_pay(handle_n_points(h), n, b.k, r.n_near);
    {
        PassArgs p;
        p.wb = r.wb;
        p.wtiles = r.wtiles;
        p.ntiles = r.nwtiles;
        p.Y = b.Y;
        p.ops = b.ops;
        p.ops_stride = b.ops_stride;
        p.img = op_image_bytes(b.k);
        p.ksteps = op_ksteps(b.k);
        p.stage_y = pass_stages_y(b.k);
        p.w_scale = r.yscale * r.yscale;
        p.Ykt = b.Ykt;
        p.Npad = r.Npad;
        p.nu = r.nu;
        p.beta = (float)(std::sqrt((double)b.k) * r.y_eps * 1.02);
        p.stages = pass_pick_stages(b.k);
        if (handle_tune(h).pass_stages >= 2) p.stages = std::min(p.stages, handle_tune(h).pass_stages);
        p.k = b.k;
        p.cert = cert_pass(n, b.k, r.b_cap);
        p.st = b.st;
        p.cand = b.cand1;
        p.cap = b.cap;
        p.pdl = handle_tune(h).pdl;
        if (tier == 5) {
            p.X = handle_x32(h);
            p.N = (int)handle_n_points(h);
            p.n = n;
            p.U32 = b.U32;
            p.KP = b.KP;
            p.U64 = b.U64;
            p.eps2 = handle_eps2(h);
            p.near = r.near;
            p.near_w = r.near_w;
            p.n_near = r.n_near;
            p.partials = b.partials;
            p.cert32 = cert_explicit(n, b.k);
        }
        if (tier == 1 && b.near_list) {
            p.N = (int)handle_n_points(h);
            if (pairs) {
                p.near = r.near;
                p.near_w = r.near_w;
                p.n_near = r.n_near;
                p.near_out = b.near_list;
                p.near_cap = (int)handle_n_points(h);
            }
            p.w32 = r.w;
            p.nb = r.Npad / T;
            p.tile0 = r.tile0;
            p.rho32 = cert_pass32(n, b.k);
        }
        handle_count_launch(h, 1, &ea, &eb);
        if (ea) cudaEventRecord(ea, s);
        RCK(launch_pass(p, restructured_pass_grid(h, b.share), s));
        if (eb) cudaEventRecord(eb, s);
        handle_push_timing(h, 1, ea, eb);
    }
    const long long pair_max = pairs ? handle_n_points(h) : -1;
    if (tier == 2 || tier == 3 || tier == 5) {
        // the explicit tier runs inside the FP64 recheck (restructured_fuse_args)
        // or (5) inside the pass
    } else if (tier == 0 || tier == 4) {
        ExplArgs x;
        x.X = handle_x32(h);
        x.N = (int)handle_n_points(h);
        x.n = n;
        x.U32 = b.U32;
        x.U32lo = b.U32lo;
        x.k = b.k;
        x.KP = b.KP;
        x.cand1 = b.cand1;
        x.cap1 = (unsigned int)b.cap;
        x.near = r.near;
        x.n_near = r.n_near;
        const bool df = tier == 4 || explicit_uses_df(n);
        x.cert = df ? cert_explicit_df(n, b.k) : cert_explicit(n, b.k);
        x.pack = tier == 4;
        x.st = b.st;
        x.cand2 = b.cand2;
        x.cap2 = b.cap;
        x.pdl = handle_tune(h).pdl;
        handle_count_launch(h, 3, &ea, &eb);
        if (ea) cudaEventRecord(ea, s);
        RCK(launch_explicit(x, df, std::max(1, handle_tune(h).expl_per_sm) * handle_sms(h), s));
        if (eb) cudaEventRecord(eb, s);
        handle_push_timing(h, 3, ea, eb);
    } else {
        // double-float Y of this basis, then the refine tier
        YdfArgs y;
        y.X = handle_x32(h);
        y.N = (int)handle_n_points(h);
        y.n = n;
        y.U32 = b.U32;
        y.U32lo = b.U32lo;
        y.KP = b.KP;
        y.Npad = r.Npad;
        y.Yh = b.Ydh;
        y.Yl = b.Ydl;
        y.KY = b.KY;
        y.st = b.st;
        y.pair_max = pair_max;
        y.cand1 = b.cand1;
        y.near_list = b.near_list;
        y.cert = cert_explicit_df(n, b.k);
        y.cand2 = reinterpret_cast<unsigned long long *>(b.cand2);
        y.cap2 = b.cap;
        RefineArgs x;
        x.pair_max = pair_max;
        x.Yh = b.Ydh;
        x.Yl = b.Ydl;
        x.Npad = r.Npad;
        x.w = r.w;
        x.nb = r.Npad / T;
        x.tile0 = r.tile0;
        x.nwt = r.nwtiles;
        x.xn = r.xn;
        x.beta = (float)(std::sqrt((double)b.k) * (df_error_unit(n) + std::ldexp(1.0, -46)) * 1.02);
        x.cand1 = b.cand1;
        x.cap1 = (unsigned int)b.cap;
        x.near = r.near;
        x.near_w = r.near_w;
        x.n_near = r.n_near;
        x.cert = cert_refine(n, b.k);
        x.st = b.st;
        x.cand2 = reinterpret_cast<unsigned long long *>(b.cand2);
        x.cap2 = b.cap;
        x.pdl = handle_tune(h).pdl;
        const int sms = handle_sms(h);
        handle_count_launch(h, 4, &ea, &eb);
        if (ea) cudaEventRecord(ea, s);
        RCK(launch_ydf_refine(y, x, b.k, 2 * sms, 0, true, s));
        if (eb) cudaEventRecord(eb, s);
        handle_push_timing(h, 4, ea, eb);
        handle_count_launch(h, 3, &ea, &eb);
        if (ea) cudaEventRecord(ea, s);
        RCK(launch_ydf_refine(y, x, b.k, 0, std::max(1, handle_tune(h).expl_per_sm) * sms, false, s));
        if (eb) cudaEventRecord(eb, s);
        handle_push_timing(h, 3, ea, eb);
    }
    return SAP_OK;
}

sap_status restructured_enqueue(sap_handle h, int share)
{
    RestrState &r = restr_state(h);
    cudaStream_t s = handle_stream(h);
    const int k = handle_k(h);
    sap_status st = restructured_enqueue_product(h, &r.gemm.tb_hi, &r.gemm.tb_lo, r.KPG, r.Y, OpsView{r.ops, &k, 1}, r.KY,
                                                 r.Ypart, handle_state(h), s, true);
    if (st != SAP_OK) return st;
    BasisView b;
    b.k = handle_k(h);
    b.KP = handle_kp(h);
    b.KY = r.KY;
    b.U32 = handle_u32(h);
    b.U32lo = handle_u32lo(h);
    b.Y = r.Y;
    b.Ykt = r.KY;
    b.ops = r.ops;
    b.ops_stride = 2 * op_image_bytes(b.k);
    b.share = share;
    b.near_list = r.near_list;
    b.Ydh = r.Ydh;
    b.Ydl = r.Ydl;
    b.st = handle_state(h);
    b.cand1 = handle_cand1(h);
    b.cand2 = handle_cand2(h);
    b.cap = handle_cap(h);
    b.U64 = handle_u64(h);
    b.partials = handle_partials(h);
    return restructured_enqueue_basis(h, b, s);
}

bool restructured_u_maps(sap_handle h, void *Uhi, void *Ulo, int KPG, CUtensorMap *mhi, CUtensorMap *mlo)
{
    RestrState &r = restr_state(h);
    const bool bf16 = handle_split_bf16(h) != 0;
    return make_map(mhi, Uhi, bf16, r.NP, KPG, KPG) && make_map(mlo, Ulo, bf16, r.NP, KPG, KPG);
}

sap_status restructured_classify(sap_handle h, int k)
{
    const RestrState &r = restr_state(h);
    if (r.k_cls == k && r.b_cap == handle_tune(h).b_cap) return SAP_OK;
    return classify(h, k);
}

sap_status restructured_project(sap_handle h, float *Y_out, int out_is_device)
{
    RestrState &r = restr_state(h);
    cudaStream_t s = handle_stream(h);
    const int k = handle_k(h);
    const int N = (int)handle_n_points(h);
    GemmArgs g = product_args(h, r);
    g.Y = r.Y;
    g.KY = r.KY;
    g.KPG = r.KPG;
    g.stages = gemm_pick_stages(r.KPG, g.nkb, r.Npad / T * g.ksplit, handle_sms(h));
    g.st = handle_state(h);
    g.Ypart = r.Ypart;
    cudaEvent_t ea, eb;
    handle_count_launch(h, 0, &ea, &eb);
    if (ea) cudaEventRecord(ea, s);
    RCK(launch_gemm_y(g, s));
    if (eb) cudaEventRecord(eb, s);
    handle_push_timing(h, 0, ea, eb);
    // Y^T (component-major) -> N x k row-major
    if (out_is_device) {
        transpose_y_kernel<<<(N * k + 255) / 256, 256, 0, s>>>(r.Y, r.KY, N, k, Y_out);
        RCK(cudaGetLastError());
        RCK(cudaStreamSynchronize(s));
    } else {
        std::vector<float> yt((size_t)r.KY * r.Npad);  // the whole block-major buffer
        RCK(cudaMemcpyAsync(yt.data(), r.Y, yt.size() * sizeof(float), cudaMemcpyDeviceToHost, s));
        RCK(cudaStreamSynchronize(s));
        for (int i = 0; i < N; ++i)
            for (int c = 0; c < k; ++c)
                Y_out[(size_t)i * k + c] = yt[(size_t)(i >> 7) * r.KY * 128 + (size_t)c * 128 + (i & 127)];
    }
    return SAP_OK;
}

sap_status restructured_project_df(sap_handle h, float *Yh_out, float *Yl_out, int out_is_device)
{
    RestrState &r = restr_state(h);
    cudaStream_t s = handle_stream(h);
    const int k = handle_k(h);
    const int N = (int)handle_n_points(h);
    YdfArgs y;
    y.X = handle_x32(h);
    y.N = N;
    y.n = handle_n_dim(h);
    y.U32 = handle_u32(h);
    y.U32lo = handle_u32lo(h);
    y.KP = handle_kp(h);
    y.Npad = r.Npad;
    y.Yh = r.Ydh;
    y.Yl = r.Ydl;
    y.KY = r.KY;
    RefineArgs unused;
    std::memset(&unused, 0, sizeof(unused));
    RCK(launch_ydf_refine(y, unused, k, 2 * handle_sms(h), 0, true, s));
    std::vector<float> th((size_t)k * r.Npad), tl((size_t)k * r.Npad);
    RCK(cudaMemcpyAsync(th.data(), r.Ydh, th.size() * sizeof(float), cudaMemcpyDeviceToHost, s));
    RCK(cudaMemcpyAsync(tl.data(), r.Ydl, tl.size() * sizeof(float), cudaMemcpyDeviceToHost, s));
    RCK(cudaStreamSynchronize(s));
    std::vector<float> oh((size_t)N * k), ol((size_t)N * k);
    for (int i = 0; i < N; ++i)
        for (int c = 0; c < k; ++c) {
            oh[(size_t)i * k + c] = th[(size_t)c * r.Npad + i];
            ol[(size_t)i * k + c] = tl[(size_t)c * r.Npad + i];
        }
    const cudaMemcpyKind kind = out_is_device ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost;
    RCK(cudaMemcpy(Yh_out, oh.data(), oh.size() * sizeof(float), kind));
    RCK(cudaMemcpy(Yl_out, ol.data(), ol.size() * sizeof(float), kind));
    return SAP_OK;
}

int restructured_tier_for(sap_handle h, int k)
{
    const int t = handle_tune(h).refine;
    const int n = handle_n_dim(h);
    if (t == 5) return k > 16 ? 0 : 5;
    if (t == 4) return 4;
    if (t == 3) return k <= 8 ? 3 : 0;
    if (t == 2) return explicit_uses_df(n) ? 0 : 2;
    if (t < 0) return n > 256 ? 1 : k <= 16 ? 5 : 0;
    return t != 0 ? 1 : 0;
}

int restructured_tier(sap_handle h) { return restructured_tier_for(h, handle_k(h)); }

// A block of the pass occupies its SM (shared memory) and spends 4-5 us on its
// start and its survivors before and after 0.7 us per tile.  Alone, a pass
// takes every SM it can use.  Passes side by side that together have more
// tiles than there are SMs take as many tiles per block as it needs for all
// their blocks to be resident at once, up to 8, past which the fixed costs no
// longer count; an excess of an eighth of the SMs is left to the first blocks
// that finish.  us per iteration with one tile per block, this rule, and 8 at
// once: 8 bases over 21 tiles each 48.7, 48.7, 54.0; 4 bases over 45 tiles
// 34.9, 31.4, 37.8; 4 over 300 tiles 55.9, 39.9, 39.9; 11 datasets of 15 tiles
// 33.3, 33.3, 39.7; 16 scenes of 500..12000 points 184, 152, 152.
int pass_share(long long tiles, int sms)
{
    return (int)std::max(1ll, std::min(8ll, (tiles + sms - 1 - sms / 8) / sms));
}

int restructured_pass_grid(sap_handle h, int share)
{
    return std::min((restr_state(h).nwtiles + share - 1) / share, handle_sms(h));
}

bool restructured_uses_refine(sap_handle h) { return restructured_tier(h) == 1; }

void restructured_fuse_args(sap_handle h, const BasisView &b, SelectUpdateArgs &u)
{
    u.fused = 0;
    u.near = nullptr;
    u.n_near = 0;
    u.cert2 = cert_explicit(handle_n_dim(h), b.k);
    const int tier = restructured_tier_for(h, b.k);
    if (tier == 5) {
        // the pass left its blocks' best pairs: one block takes the argmin
        u.pass_parts = restructured_pass_grid(h, b.share);
        u.grid = 1;
        return;
    }
    if (tier == 4) {
        // the extended tier's packed list, filtered by the final bound
        u.fused = 4;
        u.list = b.cand2;
        u.which = 2;
        u.cert2 = cert_explicit_df(handle_n_dim(h), b.k);
        return;
    }
    if (tier == 1) {
        // the refine tier's packed list: the entries are lower bounds on the
        // ratios, so the final bound itself is the threshold
        u.fused = 4;
        u.list = b.cand2;
        u.which = 2;
        u.cert2 = Cert{0.f, 0.f};
        return;
    }
    if (tier != 2 && tier != 3) return;
    RestrState &r = restr_state(h);
    u.fused = tier;
    u.near = r.near;
    u.n_near = r.n_near;
    u.list = b.cand1;
    u.which = 1;
    if (tier == 3) {
        u.cert2 = cert_explicit_df(handle_n_dim(h), b.k);
        u.grid = std::min(std::max(1, handle_tune(h).expl_per_sm) * handle_sms(h), kRecheckBlocks);
    }
}

int restructured_kernels_per_iteration(sap_handle h)
{
    // product (+ slice sum), pass, and the explicit tier, or the double-float
    // product + refine tier, or nothing (fused into the FP64 recheck or, 5,
    // into the pass)
    const int tier = restructured_tier(h);
    return 2 + (tier == 1 ? 2 : (tier == 0 || tier == 4) ? 1 : 0) + (restr_state(h).ksplit > 1 ? 1 : 0);  // 2, 3: fused
}

void restructured_free(sap_handle h)
{
    RestrState &r = restr_state(h);
    dfree(r.Xhi); dfree(r.Xlo); dfree(r.center); dfree(r.colpart); dfree(r.nu); dfree(r.w); dfree(r.wtiles);
    dfree(r.near); dfree(r.counters); dfree(r.Uhi); dfree(r.Ulo); dfree(r.Y); dfree(r.ops); dfree(r.Ypart);
    dfree(r.near_w); dfree(r.near_list); dfree(r.xn); dfree(r.Ydh); dfree(r.Ydl); dfree(r.wb);
}

void restructured_stats(sap_handle h, sap_stats *out)
{
    RestrState &r = restr_state(h);
    out->n_near = r.n_near;
    out->n_excluded = r.n_excluded;
    out->cert_bound = r.b_cap;
    out->y_error_unit = r.y_eps;
    out->ydf_error_unit = df_error_unit(handle_n_dim(h));
}

} // namespace sap
