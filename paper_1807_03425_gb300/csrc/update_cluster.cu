// update_cluster.cu -- the basis update of one SAP iteration (Algorithm 1,
// Sec. IV of Kvinge et al., arXiv:1807.03425) by a thread-block cluster, for
// FP32/BF16 data whose basis does not fit the one-row-per-thread form of
// select_update.cu (k > 8 or n > 128).
//
// The steps are those of select_update.cu's header: argmin over the blocks'
// exact results, D = x_i - x_j and c = U^T s, pivot and modified
// Gram-Schmidt in the k-dimensional coefficient space, rotation, FP64
// re-orthonormalisation, the new basis in every form the kernels read, and
// the recent argmin pairs re-evaluated as the next evaluation's bound.
//
// What bounds it, and the split.  FP64 issues at 1/64 of the FP32 rate here
// (a warp's FP64 instruction holds its SM sub-partition's pipe for about 64
// cycles), so the n k^2 / 2 FP64 products of the Gram matrix take 0.2 ms on
// one SM at n = 4096, k = 20; a dependent chain of them is no faster.  The
// rows of the basis are therefore dealt to the blocks of a cluster: the
// O(n k) and O(k^3) FP32 steps are repeated in every block (no exchange, and
// every block sees the same bits), each block forms its own rows of the
// rotated basis U' and their part of the Gram matrix G, the blocks read each
// other's parts from distributed shared memory behind one cluster barrier
// and add them in the same order, and each finishes its own rows.
//   - Modified Gram-Schmidt runs on one warp, lane m holding vector m, every
//     vector being reduced as soon as the next direction is known: the
//     operations and their order per vector are those of the sequential
//     loop, k steps deep instead of k^2 / 2.
//   - U'' = U' (I + R)^-1 = U' + U' S with |S| ~ 1e-7: U' is FP32, so its
//     product with S (as FP32 hi + lo) is formed with error-free FP32 steps,
//     accurate to 2^-46 |S| -- far below the FP64 rounding of U'' -- and two
//     FP64 additions per entry remain instead of k.
// Measured against the one-block update it replaces: 67 -> 16.5 us at n =
// 224, k = 10 (alone on the GPU); 1705 -> 129 us at n = 4096, k = 17..20,
// 1201 -> 92 us at k = 13..16 and 618 -> 66 us at k = 9..12 (averages inside
// the dimension sweep, beside the other bases' kernels, which have become
// shorter and overlap them more than when the first form took 106, 81 and 70).
#include "update_cluster.cuh"

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

namespace cg = cooperative_groups;

namespace sap {
namespace {

constexpr int UB = 256;            // threads per block
constexpr int UW = UB / 32;
constexpr int kGramRows = 64;      // rows staged in FP64 at a time
constexpr int kMaxSlices = 16;     // row slices of one Gram entry

// Blocks of the cluster: about 64 rows each, at most 16 (the largest
// cluster; beyond 8 it is a non-portable size, which this device has).
// A whole subset sweep (n = 200, k = 1..10, 25 iterations, 3 subsets) took
// 5.84 ms with 32 rows a block, 5.87 with 64, 6.01 with 128, 6.21 with 256
// and 5.95 with 16.
__host__ inline int cluster_blocks(int n)
{
    int c = 1;
    while (c < kUpdateClusterMax && c * 64 < n) c <<= 1;
    return c;
}
__host__ __device__ inline int cluster_rows(int n, int blocks) { return (n + blocks - 1) / blocks; }

// Shared memory of one block (dynamic).
template <int K>
struct UpdLayout {
    static constexpr int KS = K | 1;                   // odd row stride
    static constexpr int KK = K * K;
    static constexpr int E = K * (K + 1) / 2;
    // doubles first
    static constexpr size_t o_gpart = 0;                                // E: this block's Gram sums
    static constexpr size_t o_slice = o_gpart + 8 * (size_t)E;          // UB
    static constexpr size_t o_G = o_slice + 8 * (size_t)UB;             // KK
    static constexpr size_t o_Ri = o_G + 8 * (size_t)KK;                // KK
    static constexpr size_t o_stage = o_Ri + 8 * (size_t)KK;            // kGramRows x (K + 1)
    static constexpr size_t o_rd = o_stage + 8 * (size_t)kGramRows * (K + 1);  // K
    static constexpr size_t o_seedp = o_rd + 8 * (size_t)K;             // floats: kWatch x (K + 1)
    static constexpr size_t o_S1 = o_seedp + 4 * (size_t)kWatch * (K + 1);
    static constexpr size_t o_R2 = o_S1 + 4 * (size_t)KK;
    static constexpr size_t o_Sq = o_R2 + 4 * (size_t)KK;
    static constexpr size_t o_Shi = o_Sq + 4 * (size_t)KK;
    static constexpr size_t o_Slo = o_Shi + 4 * (size_t)KK;
    static constexpr size_t o_Q = o_Slo + 4 * (size_t)KK;               // [m][q]
    static constexpr size_t o_rows = o_Q + 4 * (size_t)KK;              // rows x KS
    static size_t bytes(int rows) { return o_rows + 4 * (size_t)rows * KS; }
};

template <int K>
__global__ void __launch_bounds__(UB, 1) update_cluster_kernel(SelectUpdateArgs a, int nparts)
{
    using Lay = UpdLayout<K>;
    constexpr int KS = Lay::KS, KP4 = (K + 3) / 4 * 4;
    extern __shared__ __align__(16) unsigned char smb[];
    double *gpart = reinterpret_cast<double *>(smb + Lay::o_gpart);
    double *slice = reinterpret_cast<double *>(smb + Lay::o_slice);
    double *G = reinterpret_cast<double *>(smb + Lay::o_G);
    double *Ri = reinterpret_cast<double *>(smb + Lay::o_Ri);
    double *stage = reinterpret_cast<double *>(smb + Lay::o_stage);
    double *Rd = reinterpret_cast<double *>(smb + Lay::o_rd);
    float *seedp = reinterpret_cast<float *>(smb + Lay::o_seedp);
    float *S1 = reinterpret_cast<float *>(smb + Lay::o_S1);
    float *R2 = reinterpret_cast<float *>(smb + Lay::o_R2);
    float *Sq = reinterpret_cast<float *>(smb + Lay::o_Sq);
    float *Shi = reinterpret_cast<float *>(smb + Lay::o_Shi);
    float *Slo = reinterpret_cast<float *>(smb + Lay::o_Slo);
    float *Qs = reinterpret_cast<float *>(smb + Lay::o_Q);
    float *rows = reinterpret_cast<float *>(smb + Lay::o_rows);
    __shared__ float red[UW * (K + 1)];
    __shared__ float cvec[K + 1], cw[K], qd[K + 1];
    __shared__ Partial best_sh;
    __shared__ int2 watch[kWatch];
    __shared__ int watch_n, watch_pos, iter, hist_cap, cnt1, cnt2, alive0_sh;
    __shared__ float av_sh, asd_sh, d_sh;
    __shared__ float seed_sh[kWatch];

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n = a.n, kk = a.k;
    ProbState *st = a.st;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), C = (int)cluster.num_blocks();
    const int R = cluster_rows(n, C), l0 = rank * R, nr = max(0, min(R, n - l0));

    // Programmatic launch: the next product may start its prologue (it waits
    // for this kernel before it reads the basis).
    grid_dep_launch();
    grid_dep_wait();

    // ---- 1. argmin over the blocks' results (every block of the cluster)
    if (w == 0) {
        Partial b = {INFINITY, 0x7fffffff, 0x7fffffff};
        for (int p0 = 0; p0 < nparts; p0 += 256) {
            long long rq[8], ij[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int p = p0 + lane + 32 * u;
                const long long *src = reinterpret_cast<const long long *>(a.partials + (p < nparts ? p : 0));
                rq[u] = __ldcg(src);
                ij[u] = __ldcg(src + 1);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (p0 + lane + 32 * u >= nparts) break;
                const Partial q = {__longlong_as_double(rq[u]), (int)(ij[u] & 0xffffffff), (int)(ij[u] >> 32)};
                if (better_q(q.r, q.i, q.j, b.r, b.i, b.j)) b = q;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            Partial q;
            q.r = __shfl_xor_sync(0xffffffffu, b.r, o);
            q.i = __shfl_xor_sync(0xffffffffu, b.i, o);
            q.j = __shfl_xor_sync(0xffffffffu, b.j, o);
            if (better_q(q.r, q.i, q.j, b.r, b.i, b.j)) b = q;
        }
        if (lane == 0) best_sh = b;
    } else if (w == 1) {
        if (lane == 0) {
            iter = st->iter;
            hist_cap = st->hist_cap;
            cnt1 = st->cnt1;
            cnt2 = st->cnt2;
            watch_n = st->watch_n;
            watch_pos = st->watch_pos;
        }
        if (lane < kWatch) watch[lane] = st->watch[lane];
    }
    __syncthreads();
    const Partial b = best_sh;
    const bool none = !(b.r < INFINITY);  // the same in every block

    // Records the result (history, state): one thread of block 0, after the
    // cluster's first barrier, when every block has read the state it needs.
    auto record = [&]() {
        const double r = none ? b.r : sqrt(b.r);
        if (!none) {
            // whether the seed bound this evaluation started from was tight
            const float sd = __uint_as_float(st->seed_ub);
            st->seed_miss = sd <= (float)r * 1.01f ? 0 : min(st->seed_miss + 1, 1 << 20);
        } else {
            atomicOr(&st->status, ST_NO_SECANT);
        }
        if (iter < hist_cap) {
            a.hist[iter] = none ? __longlong_as_double(0x7ff8000000000000ll) : r;
            a.argmin[iter] = none ? make_int2(-1, -1) : make_int2(b.i, b.j);
        }
        st->iter = iter + 1;
        st->last_r = r;
        st->last_i = none ? -1 : b.i;
        st->last_j = none ? -1 : b.j;
        st->last_cnt1 = cnt1;
        st->last_cnt2 = cnt2;
        st->cnt1 = 0;
        st->tile_next = 0;
        st->cnt2 = 0;
        st->cntn = 0;
        st->ticket = 0;
        st->run_ub1 = 0x7f800000u;
        st->run_ub2 = 0x7f800000u;
    };
    if (none) {
        if (tid == 0 && rank == 0) record();
        return;
    }
    // the watch list with the new pair, in every block's copy
    if (tid == 0) {
        bool present = false;
        for (int q = 0; q < watch_n; ++q) present |= (watch[q].x == b.i && watch[q].y == b.j);
        if (!present) {
            watch[watch_pos] = make_int2(b.i, b.j);
            watch_pos = (watch_pos + 1) % kWatch;
            if (watch_n < kWatch) ++watch_n;
        }
    }

    // ---- 2. D = x_i - x_j, |D|^2 and U^T D: every block over all rows,
    // thread t the rows t, t + 256, ... (FP32)
    const float *X = static_cast<const float *>(a.X);
    const float *xi = X + (size_t)b.i * n, *xj = X + (size_t)b.j * n;
    {
        float v[K + 1];
#pragma unroll
        for (int q = 0; q <= K; ++q) v[q] = 0.f;
#pragma unroll 2
        for (int l = tid; l < n; l += UB) {
            const float D = xi[l] - xj[l];
            float u[KP4];
#pragma unroll
            for (int c = 0; c < KP4; c += 4) {
                const float4 t = __ldcg(reinterpret_cast<const float4 *>(a.U32 + (size_t)l * a.KP + c));
                u[c] = t.x; u[c + 1] = t.y; u[c + 2] = t.z; u[c + 3] = t.w;
            }
            v[K] = fmaf(D, D, v[K]);
#pragma unroll
            for (int c = 0; c < K; ++c) v[c] = fmaf(u[c], D, v[c]);
        }
        warp_sum_multi<float, K + 1>(v);
        if (lane == 0)
#pragma unroll
            for (int q = 0; q <= K; ++q) red[w * (K + 1) + q] = v[q];
        __syncthreads();
        if (tid <= K) {
            float s = 0.f;
            for (int p = 0; p < UW; ++p) s += red[p * (K + 1) + tid];
            cvec[tid] = s;
        }
        __syncthreads();
    }

    // ---- 3-4. pivot, modified Gram-Schmidt on [c, e_l (l != t)] and the
    // rotation coefficients: warp 0, lane m holding vector m
    // (a direction travels from its lane through shared memory: as K shuffles
    // per step this section took 42 K of the kernel's 71 K cycles at n = 200,
    // k = 10; now 17 K)
    if (w == 0) {
        const float d = sqrtf(cvec[K]);
        if (lane < K) cw[lane] = lane < kk ? cvec[lane] / d : 0.f;
        __syncwarp();
        float x[K], r2 = 0.f, cmax = -1.f;
        int t = 0;
#pragma unroll
        for (int q = 0; q < K; ++q) {
            x[q] = cw[q];
            r2 = fmaf(x[q], x[q], r2);
            if (q < kk && fabsf(x[q]) > cmax) { cmax = fabsf(x[q]); t = q; }
        }
        if (lane != 0) {
            const int lm = (lane - 1) < t ? (lane - 1) : lane;  // list entry m >= 1 is column lm
#pragma unroll
            for (int q = 0; q < K; ++q) x[q] = q == lm ? 1.f : 0.f;
        }
#pragma unroll 1
        for (int p = 0; p < kk; ++p) {
            if (lane == p) {
                float nn = 0.f;
#pragma unroll
                for (int q = 0; q < K; ++q) nn = fmaf(x[q], x[q], nn);
                const bool alive = nn > 0.f;
                const float inv = alive ? 1.f / sqrtf(nn) : 0.f;
#pragma unroll
                for (int q = 0; q < K; ++q) qd[q] = x[q] = x[q] * inv;
                qd[K] = alive ? 1.f : 0.f;
                if (p == 0) alive0_sh = alive ? 1 : 0;
            }
            __syncwarp();
            float qp[K], h = 0.f;
#pragma unroll
            for (int q = 0; q < K; ++q) qp[q] = qd[q];
            const bool alive = qd[K] != 0.f;  // the same in every lane
            __syncwarp();                     // read before the next step writes
            if (!alive) continue;
#pragma unroll
            for (int q = 0; q < K; ++q) h = fmaf(qp[q], x[q], h);
            if (lane > p)
#pragma unroll
                for (int q = 0; q < K; ++q) x[q] = fmaf(-h, qp[q], x[q]);
        }
        if (lane < K)
#pragma unroll
            for (int q = 0; q < K; ++q) Qs[lane * K + q] = lane < kk ? x[q] : 0.f;
        if (lane == 0) {
            const float al = (float)a.alpha;
            float av, as;
            if (a.mode == 1) {  // angle reading
                const float nv = sqrtf(r2);
                const float ne = sqrtf(r2 < 1.f ? 1.f - r2 : 0.f);
                av = (nv > 0.f ? (1.f - al) / nv : 0.f) - (ne > 0.f ? al / ne : 0.f);
                as = ne > 0.f ? al / ne : 0.f;
            } else {            // literal reading: (1-a) v + a (s - v)
                av = 1.f - 2.f * al;
                as = al;
            }
            av_sh = av;
            asd_sh = as / d;  // applied to D = d s
            d_sh = d;
        }
    }
    __syncthreads();

    // ---- the block's rows of U' and their part of the Gram matrix
    const int E = kk * (kk + 1) / 2;
    const int slices = E <= UB ? min(kMaxSlices, UB / E) : 1;
    constexpr int NE = (Lay::E + UB - 1) / UB;  // entries per thread when E > UB
    int ep[NE], eq[NE];
    const int ne = E <= UB ? 1 : (E - tid + UB - 1) / UB;  // entries of this thread
    {
        const int e0 = E <= UB ? tid % E : tid;
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            int e = e0 + i * UB, p = 0;
            if (e >= E) e = 0;
            while (e >= kk - p) { e -= kk - p; ++p; }
            ep[i] = p;
            eq[i] = p + e;
        }
    }
    const int sl = E <= UB ? tid / E : 0;  // row slice; threads past the last one idle
    double inv0 = 0.0;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        // column 0 = av U c + as s (its length comes out of the Gram matrix
        // below), column m >= 1 = U q_m.  Second pass: the direction
        // vanished (alpha = 1 with s in the span); q_0 in place of column 0,
        // s itself when P P^T s = 0
        const float av = av_sh, asd = asd_sh;
#pragma unroll 1
        for (int r = tid; r < nr; r += UB) {
            const int l = l0 + r;
            const float D = xi[l] - xj[l];
            float u[KP4];
#pragma unroll
            for (int c = 0; c < KP4; c += 4) {
                const float4 t = __ldcg(reinterpret_cast<const float4 *>(a.U32 + (size_t)l * a.KP + c));
                u[c] = t.x; u[c + 1] = t.y; u[c + 2] = t.z; u[c + 3] = t.w;
            }
            float *row = rows + (size_t)r * KS;
            if (pass == 0) {
                float v0 = 0.f;
#pragma unroll
                for (int c = 0; c < K; ++c) v0 = fmaf(u[c], cw[c], v0);
                row[0] = fmaf(av, v0, asd * D);
            } else {
                float q1 = 0.f;
#pragma unroll
                for (int c = 0; c < K; ++c) q1 = fmaf(u[c], Qs[c], q1);
                row[0] = alive0_sh ? q1 : D / d_sh;
            }
#pragma unroll(K <= 8 ? K : 4)
            for (int m = 1; m < kk; ++m) {
                float s = 0.f;
#pragma unroll
                for (int c = 0; c < K; ++c) s = fmaf(u[c], Qs[m * K + c], s);
                row[m] = s;
            }
        }
        double acc[NE];
#pragma unroll
        for (int i = 0; i < NE; ++i) acc[i] = 0.0;
        for (int r0 = 0; r0 < nr; r0 += kGramRows) {
            const int rc = min(kGramRows, nr - r0);
            __syncthreads();  // rows written; the previous chunk has been read
            for (int idx = tid; idx < rc * kk; idx += UB) {
                const int r = idx / kk, m = idx % kk;
                stage[r * (K + 1) + m] = widen(rows[(size_t)(r0 + r) * KS + m]);
            }
            __syncthreads();
            if (sl < slices)
                for (int r = sl; r < rc; r += slices) {
                    const double *sr = stage + r * (K + 1);
#pragma unroll
                    for (int i = 0; i < NE; ++i)
                        if (i < ne) acc[i] = fma(sr[ep[i]], sr[eq[i]], acc[i]);
                }
        }
        if (E <= UB) {
            if (slices > 1) {
                slice[tid] = acc[0];
                __syncthreads();
                if (tid < E) {
                    double s = acc[0];
                    for (int q = 1; q < slices; ++q) s += slice[q * E + tid];
                    gpart[tid] = s;
                }
            } else if (tid < E) {
                gpart[tid] = acc[0];
            }
        } else {
#pragma unroll
            for (int i = 0; i < NE; ++i)
                if (tid + i * UB < E) gpart[tid + i * UB] = acc[i];
        }
        cluster.sync();
        // the blocks' parts, added in the same order everywhere (two
        // accumulators: half the dependent FP64 additions)
        for (int e = tid; e < E; e += UB) {
            double s0 = 0.0, s1 = 0.0;
            for (int q = 0; q < C; q += 2) {
                s0 += *cluster.map_shared_rank(gpart + e, q);
                if (q + 1 < C) s1 += *cluster.map_shared_rank(gpart + e, q + 1);
            }
            int p = 0, f = e;
            while (f >= kk - p) { f -= kk - p; ++p; }
            G[p * K + p + f] = s0 + s1;
        }
        __syncthreads();
        const double g00 = G[0];
        if (g00 > 0.0) {
            inv0 = rsqrt_scale(g00);  // any scale near 1/|u'_0| gives the same basis
            break;
        }
        cluster.sync();  // every block has read the parts: the second pass rewrites them
        if (pass == 1) inv0 = 0.0;  // no direction at all (not reached with orthonormal U)
    }
    if (rank == 0 && tid == UB - 32) {
        record();
        for (int q = 0; q < kWatch; ++q) st->watch[q] = watch[q];
        st->watch_n = watch_n;
        st->watch_pos = watch_pos;
        if (a.seeds_in_product) st->seed_ub = 0x7f800000u;  // the next product merges its seeds into +inf
    }

    // ---- 5. S = (I + R)^-1 - I with G = (I + R)^T (I + R), column 0 scaled.
    // Series in E = G - I to third order when max|E| <= 1e-5 sqrt(8 / k): R =
    // R1 + R2 + R3, R1 = triu(E) with halved diagonal (FP64), R2 = split of
    // -R1^T R1, R3 = split of -(R1^T R2 + R2^T R1) (split: upper triangle,
    // halved diagonal), (I + R)^-1 = I - R1 - R2 - R3 + R1^2 + R1 R2 + R2 R1
    // - R1^3.  Terms past R1 are at most k max|E|^2 = 8e-10 and are
    // evaluated in FP32 (error 5e-17); the truncation is (8e-10)^2.  Else a
    // Cholesky factorisation.
    const float lim = K <= 8 ? 1e-5f : 1e-5f * sqrtf(8.f / K);
    bool small = true;
    for (int e = tid; e < K * K; e += UB) {
        const int p = e / K, q = e % K;
        double v = 0.0;
        if (q >= p && q < kk) {
            v = G[p * K + q];
            if (p == 0) v *= q == 0 ? inv0 * inv0 : inv0;
            if (p == q) v -= 1.0;
            if (fabs(v) > (double)lim) small = false;
            if (p == q) v *= 0.5;
        }
        Ri[e] = v;       // R1
        S1[e] = (float)v;
    }
    small = __syncthreads_and(small ? 1 : 0) != 0;
    if (small) {
        for (int e = tid; e < K * K; e += UB) {
            const int p = e / K, q = e % K;
            float tt = 0.f, sq = 0.f;
            if (q >= p && q < kk) {
                for (int m = 0; m <= p; ++m) tt = fmaf(S1[m * K + p], S1[m * K + q], tt);  // (R1^T R1)_pq
                for (int m = p; m <= q; ++m) sq = fmaf(S1[p * K + m], S1[m * K + q], sq);  // (R1^2)_pq
            }
            R2[e] = q > p ? -tt : (q == p ? -0.5f * tt : 0.f);
            Sq[e] = sq;
        }
        __syncthreads();
        for (int e = tid; e < K * K; e += UB) {
            const int p = e / K, q = e % K;
            if (q < p || q >= kk) continue;
            float m3 = 0.f, r12 = 0.f, r21 = 0.f, r13 = 0.f;
            for (int m = 0; m <= p; ++m) {
                m3 = fmaf(S1[m * K + p], R2[m * K + q], m3);
                m3 = fmaf(R2[m * K + p], S1[m * K + q], m3);
            }
            for (int m = p; m <= q; ++m) {
                r12 = fmaf(S1[p * K + m], R2[m * K + q], r12);  // (R1 R2)_pq
                r21 = fmaf(R2[p * K + m], S1[m * K + q], r21);  // (R2 R1)_pq
                r13 = fmaf(Sq[p * K + m], S1[m * K + q], r13);  // (R1^3)_pq
            }
            const float r3 = q > p ? -m3 : -0.5f * m3;
            const float hi = -R2[e] - r3 + Sq[e] + r12 + r21 - r13;
            double s = -Ri[e] + (double)hi;
            if (p == 0) s = q == 0 ? (1.0 + s) * inv0 : s * inv0;
            G[e] = s;  // entry (0, 0): the full factor of column 0
            const float sh = (float)s;
            Shi[e] = sh;
            Slo[e] = (float)(s - (double)sh);
        }
    } else {
        // G = I + E with the scaled column 0, right-looking Cholesky on the
        // upper triangle (lane m owns column m), then the inverse by back
        // substitution
        __syncthreads();
        if (w == 0) {
            if (lane < kk) G[lane] *= lane == 0 ? inv0 * inv0 : inv0;
            __syncwarp();
            double rinv_own = 0.0;
#pragma unroll 1
            for (int j = 0; j < kk; ++j) {
                const double gjj = G[j * K + j];
                const double rinv = rsqrt(gjj);
                __syncwarp();
                if (lane == j) { G[j * K + j] = gjj * rinv; rinv_own = rinv; }
                if (lane > j && lane < kk) G[j * K + lane] *= rinv;
                __syncwarp();
                if (lane > j && lane < kk)
                    for (int p = j + 1; p <= lane; ++p)
                        G[p * K + lane] = fma(-G[j * K + p], G[j * K + lane], G[p * K + lane]);
                __syncwarp();
            }
            if (lane < kk) Rd[lane] = rinv_own;
            __syncwarp();
            if (lane < kk) {
                for (int i = 0; i < kk; ++i) Ri[i * K + lane] = 0.0;
#pragma unroll 1
                for (int i = lane; i >= 0; --i) {
                    double s = (i == lane) ? 1.0 : 0.0;
                    for (int p = i + 1; p <= lane; ++p) s = fma(-G[i * K + p], Ri[p * K + lane], s);
                    Ri[i * K + lane] = s * Rd[i];
                }
                Ri[lane] *= inv0;
            }
        }
    }
    __syncthreads();

    // ---- 6. the block's rows of U'', in every form the kernels read
    // (one entry per thread and turn, lanes over rows: a row per thread left
    // most threads idle, 12.6 K cycles at n = 200, k = 10; now 2.4 K)
    const double s00 = small ? G[0] : 0.0;
#pragma unroll 1
    for (int e = tid; e < nr * kk; e += UB) {
        const int m = e / nr, r = e - m * nr, l = l0 + r;
        const float *row = rows + (size_t)r * KS;
        double s;
        float hi = 0.f, rest = 0.f;  // x_m + correction as an FP32 pair (when available)
        if (small && m > 0) {
            // x_m + sum_p x_p S_pm: two chains of error-free steps
            float h0 = 0.f, e0 = 0.f, h1 = 0.f, e1 = 0.f;
#pragma unroll 2
            for (int p = 0; p <= m; p += 2) {
                xs_fma(h0, e0, row[p], Shi[p * K + m], Slo[p * K + m]);
                if (p + 1 <= m) xs_fma(h1, e1, row[p + 1], Shi[(p + 1) * K + m], Slo[(p + 1) * K + m]);
            }
            float hs, es;
            xs_two_sum(h0, h1, hs, es);
            es = __fadd_rn(es, __fadd_rn(e0, e1));
            s = widen(row[m]) + (widen(hs) + widen(es));
            xs_two_sum(row[m], hs, hi, rest);
            rest = __fadd_rn(rest, es);
        } else if (small) {
            s = widen(row[0]) * s00;
        } else {
            s = 0.0;
            for (int p = 0; p <= m; ++p) s = fma(widen(row[p]), Ri[p * K + m], s);
        }
        a.U64[(size_t)m * n + l] = s;
        const float sf = (float)s;
        a.U32[(size_t)l * a.KP + m] = sf;
        // the residual from the FP32 pair where sf is its high part (FP64
        // operations are the scarce resource here)
        if (a.U32lo) a.U32lo[(size_t)l * a.KP + m] = (small && m > 0 && sf == hi) ? rest : (float)(s - (double)sf);
        if (a.Uhi) {
            // hi + lo * 2^-s of the FP32 value (the FP32 rounding adds 2^-24
            // relative to the split residual)
            const size_t idx = (size_t)m * a.NP + l;
            if (a.split_bf16) {
                const __nv_bfloat16 h = __float2bfloat16_rn(sf);
                static_cast<__nv_bfloat16 *>(a.Uhi)[idx] = h;
                static_cast<__nv_bfloat16 *>(a.Ulo)[idx] =
                    __float2bfloat16_rn((sf - __bfloat162float(h)) * a.split_scale);
            } else {
                const __half h = __float2half_rn(sf);
                static_cast<__half *>(a.Uhi)[idx] = h;
                static_cast<__half *>(a.Ulo)[idx] = __float2half_rn((sf - __half2float(h)) * a.split_scale);
            }
        }
    }
    if (a.seeds_in_product) {
        cluster.sync();  // no block leaves while another reads its parts
        return;
    }

    // ---- seeds: the recent argmin pairs under the new basis, warp w pair w
    // over the block's rows, the blocks' sums added by block 0
    __syncthreads();
    const int nwatch = watch_n;
    if (w < nwatch) {
        float v[K + 1];
#pragma unroll
        for (int q = 0; q <= K; ++q) v[q] = 0.f;
        const int2 pr = watch[w];
        if (SAP_PAIR_OK(st, pr, a.N)) {
            const float *wi = X + (size_t)pr.x * n + l0, *wj = X + (size_t)pr.y * n + l0;
            for (int r = lane; r < nr; r += 32) {
                const float D = wi[r] - wj[r];
                const float *row = a.U32 + (size_t)(l0 + r) * a.KP;  // written by this block above
                v[K] = fmaf(D, D, v[K]);
#pragma unroll
                for (int c = 0; c < KP4; c += 4) {
                    const float4 u = __ldcg(reinterpret_cast<const float4 *>(row + c));
                    v[c] = fmaf(u.x, D, v[c]);
                    if (c + 1 < K) v[c + 1 < K ? c + 1 : 0] = fmaf(u.y, D, v[c + 1 < K ? c + 1 : 0]);
                    if (c + 2 < K) v[c + 2 < K ? c + 2 : 0] = fmaf(u.z, D, v[c + 2 < K ? c + 2 : 0]);
                    if (c + 3 < K) v[c + 3 < K ? c + 3 : 0] = fmaf(u.w, D, v[c + 3 < K ? c + 3 : 0]);
                }
            }
        }
        warp_sum_multi<float, K + 1>(v);
        if (lane == 0)
#pragma unroll
            for (int q = 0; q <= K; ++q) seedp[w * (K + 1) + q] = v[q];
    }
    cluster.sync();
    if (rank == 0 && w < nwatch) {
        float zz = 0.f, dd = 0.f;
        if (lane <= K) {  // lanes past 31 do not exist: K = 32's length sum below
            float s = 0.f;
            for (int q = 0; q < C; ++q) s += *cluster.map_shared_rank(seedp + w * (K + 1) + lane, q);
            if (lane < K) zz = s * s;
            else dd = s;
        }
        if (K == 32) {
            for (int q = 0; q < C; ++q) dd += *cluster.map_shared_rank(seedp + w * (K + 1) + K, q);
        } else {
            dd = __shfl_sync(0xffffffffu, dd, K % 32);
        }
        zz = warp_sumf(zz);
        if (lane == 0) seed_sh[w] = dd > 1e-30f ? cert_upper(sqrtf(zz / dd), a.seed_cert) : INFINITY;
    }
    __syncthreads();
    if (rank == 0 && tid == 0) {
        float m = INFINITY;
        for (int q = 0; q < nwatch; ++q) m = fminf(m, seed_sh[q]);
        st->seed_ub = __float_as_uint(m);
    }
    cluster.sync();  // no block leaves while block 0 reads its sums
}

template <int K>
cudaError_t configure_k()
{
    cudaError_t e = cudaFuncSetAttribute(update_cluster_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)UpdLayout<K>::bytes(cluster_rows(16384, kUpdateClusterMax)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(update_cluster_kernel<K>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <int K>
cudaError_t launch_k(const SelectUpdateArgs &a, int nparts, cudaStream_t s)
{
    const int C = cluster_blocks(a.n);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(UB);
    cfg.dynamicSmemBytes = UpdLayout<K>::bytes(cluster_rows(a.n, C));
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = a.pdl ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, update_cluster_kernel<K>, a, nparts);
}

} // namespace

cudaError_t update_cluster_configure()
{
    cudaError_t e = cudaSuccess;
    auto f = [&](cudaError_t x) { if (x != cudaSuccess) e = x; };
    f(configure_k<1>()); f(configure_k<2>()); f(configure_k<3>()); f(configure_k<4>());
    f(configure_k<5>()); f(configure_k<6>()); f(configure_k<7>()); f(configure_k<8>());
    f(configure_k<12>()); f(configure_k<16>()); f(configure_k<24>()); f(configure_k<32>());
    return e;
}

cudaError_t launch_update_cluster(const SelectUpdateArgs &a, int nparts, cudaStream_t s)
{
    switch (a.k) {
    case 1: return launch_k<1>(a, nparts, s);
    case 2: return launch_k<2>(a, nparts, s);
    case 3: return launch_k<3>(a, nparts, s);
    case 4: return launch_k<4>(a, nparts, s);
    case 5: return launch_k<5>(a, nparts, s);
    case 6: return launch_k<6>(a, nparts, s);
    case 7: return launch_k<7>(a, nparts, s);
    case 8: return launch_k<8>(a, nparts, s);
    default: break;
    }
    if (a.k <= 12) return launch_k<12>(a, nparts, s);
    if (a.k <= 16) return launch_k<16>(a, nparts, s);
    if (a.k <= 24) return launch_k<24>(a, nparts, s);
    return launch_k<32>(a, nparts, s);
}

} // namespace sap
