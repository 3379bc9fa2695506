// gemm_tc.cuh -- launcher interface of the tensor-core product Y = X U.
#pragma once

#include <cuda.h>
#include "sap_internal.cuh"

namespace sap {

// Operands of the all-pairs filter.  For a pair, |y_i - y_j|^2 = s_i + s_j -
// 2 <y_i, y_j> is one contraction of K-axis vectors
//     A_i = [h_i, h_i, l_i | s_i', 1],   B_j = -2 [h_j, l_j, h_j | ...] resp. [.. | 1, s_j'],
// with y (scaled by a power of two to |y| <= 64) = h + l in two FP16 terms and
// s' = (1 - kappa) |y|^2 - kabs / 2 in two FP16 terms: kappa and kabs bound
// every error of the contraction, so the result is a certified lower bound of
// |y_i - y_j|^2 (op_bounds).  Four components take three 4-element halves
// (8 bytes) of the K axis, the norms one.  An image holds 128 rows in the
// unswizzled K-major core-matrix order of the MMA: [K / 8][row / 8][row % 8][8
// elements]; a block's A image is followed by its B image.
struct OpGroup {
    uint32_t off;      // the basis's A image within a block's images
    uint32_t img;      // bytes of one image
    int g;             // group of 4 components within the basis; -1: padding
    int last;          // the basis's last group: writes the norms
    float keep, kabs2; // 1 - kappa, kabs / 2
};
constexpr int kMaxOpGroups = 64;   // 256 components
constexpr int kMaxOpBases = 20;
__host__ __device__ inline int op_ksteps(int k) { return ((3 * ((k + 3) / 4) + 1) * 4 + 15) / 16; }  // K / 16
__host__ __device__ inline uint32_t op_image_bytes(int k) { return (uint32_t)op_ksteps(k) * 4096u; }

struct GemmArgs {
    CUtensorMap ta_hi, ta_lo;   // X split parts: Npad x NP, 16-bit, box 64 x 128
    CUtensorMap tb_hi, tb_lo;   // U split parts: KPG x NP, 16-bit, box 64 x KPG
    float *Y;                   // FP32, block-major: [Npad/128][KY][128]
    // optional: the rows of Y as operands of the all-pairs pass's tensor-core
    // filter (see OpGroup), for `nbases` bases whose components follow one
    // another in Y; block b's images start at ops + b * ops_stride
    unsigned char *ops = nullptr;
    uint32_t ops_stride = 0;
    int nbases = 0;
    int base_group[kMaxOpBases + 1];    // first group of 4 components of each basis, and the end
    OpGroup groups[kMaxOpGroups];
    float ops_scale = 1.f;              // power of two: |y| * ops_scale <= 64
    int KY;                     // components written (multiple of 4, <= KPG)
    int Npad;                   // rows (multiple of 128)
    int nkb;                    // K blocks of 64
    int KPG;                    // MMA N: multiple of 16, 16..256
    int ab_bf16;                // operand type: 1 BF16, 0 FP16
    int stages;                 // shared-memory ring depth
    float lo_scale;             // 2^-s: weight of the low-part accumulator
    float out_scale;            // 1/scale of X
    ProbState *st;              // receives ST_TIMEOUT if a wait gives up
    int ksplit;                 // K slices (grid.y); > 1: raw slices go to Ypart
    float *Ypart;               // ksplit x KY x Npad FP32 (ksplit > 1)
    int pdl;                    // programmatic launch (see sap_internal.cuh)
    // Seeds of the next all-pairs pass, computed by idle warps of every CTA
    // (single-basis handles; null seed_st: none): the recent argmin pairs'
    // ratios under the basis this product uses, in extended precision from
    // explicit differences, as certified upper bounds merged into
    // seed_st->seed_ub by an atomic minimum (the update that changed the
    // basis reset it to +inf; an unchanged basis keeps its valid bound).
    const float *seed_X = nullptr;   // N x n row-major FP32 points
    const float *seed_U = nullptr;   // the basis, FP32 n x KP row-major ...
    const float *seed_Ulo = nullptr; // ... and its FP32 residual
    ProbState *seed_st = nullptr;
    int seed_N = 0, seed_n = 0, seed_k = 0, seed_KP = 0;
};

size_t gemm_smem_bytes(int KPG, int stages);
int gemm_pick_stages(int KPG, int nkb, int ctas, int sms);
cudaError_t gemm_configure();
// Y = X U; with ksplit > 1 each K slice accumulates separately (shorter FP32
// chains) and a second kernel sums the slices into Y.
cudaError_t launch_gemm_y(const GemmArgs &a, cudaStream_t s);

} // namespace sap
