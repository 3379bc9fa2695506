// basis_forms.cu -- the small transfers around a run: a new basis in every
// form the kernels read, and the results of a run gathered for one copy.
//
// A basis arrives as n x k FP64; the kernels read it as FP64 column-major,
// FP32 row-major with its FP32 residual, and split 16-bit operands.  All of
// them are formed on the device from one upload: five pageable copies (and
// the host loops before them) took 100 us per call at n = 100, k = 5 and 11
// ms for the 210 columns of a sweep at n = 4096; one copy and one launch
// replace them.  Likewise the histories, pairs and status words of a run
// come back in one copy instead of three per dataset.  What bounds these
// kernels is their launch (a few us, under 1 MB moved).
#include "basis_forms.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace sap {
namespace {

// blockIdx.y: basis; thread: one coordinate l.  Pad rows and columns of the
// destinations were cleared when they were allocated.
__global__ void __launch_bounds__(128) basis_forms_kernel(const double *src, int n, const __grid_constant__ BasisFormsArgs a)
{
    const BasisForms &b = a.b[blockIdx.y];
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l == 0 && b.st) {
        ProbState p = {};
        p.seed_ub = p.run_ub1 = p.run_ub2 = 0x7f800000u;
        p.hist_cap = a.hist_cap;
        p.last_r = INFINITY;
        p.last_i = p.last_j = -1;
        *b.st = p;
    }
    if (l >= n) return;
    for (int c = 0; c < b.k; ++c) {
        const double v = src[(size_t)c * n + l];
        if (b.U64 != src) b.U64[(size_t)c * n + l] = v;
        const float f = (float)v;
        b.U32[(size_t)l * b.KP + c] = f;
        b.U32lo[(size_t)l * b.KP + c] = (float)(v - (double)f);
        if (!b.Uhi) continue;
        const size_t idx = (size_t)c * b.NP + l;
        if (a.bf16) {
            const __nv_bfloat16 h = __double2bfloat16(v);
            static_cast<__nv_bfloat16 *>(b.Uhi)[idx] = h;
            static_cast<__nv_bfloat16 *>(b.Ulo)[idx] = __double2bfloat16((v - (double)__bfloat162float(h)) * 256.0);
        } else {
            const __half h = __double2half(v);
            static_cast<__half *>(b.Uhi)[idx] = h;
            static_cast<__half *>(b.Ulo)[idx] = __double2half((v - (double)__half2float(h)) * 2048.0);
        }
    }
}

// out: count status words, count x cnt ratios, count x cnt pairs, all 64-bit
// (pairs as two words); blockIdx.x: problem.  Status words are cleared.
__global__ void __launch_bounds__(128) gather_kernel(const RunView *views, RunView one, int cnt, int with_pairs,
                                                     long long *out)
{
    const int q = blockIdx.x, count = gridDim.x;
    const RunView v = views ? views[q] : one;
    if (threadIdx.x == 0) {
        out[q] = v.st->status;
        v.st->status = 0;
    }
    double *hist = reinterpret_cast<double *>(out + count) + (size_t)q * cnt;
    long long *am = out + count + (size_t)count * cnt + 2 * (size_t)q * cnt;
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        hist[t] = v.hist[t];
        if (with_pairs) {
            const int2 p = v.am[t];
            am[2 * t] = p.x;
            am[2 * t + 1] = p.y;
        }
    }
}

} // namespace

cudaError_t launch_basis_forms(const double *src, int n, const BasisFormsArgs &a, int count, cudaStream_t s)
{
    basis_forms_kernel<<<dim3((n + 127) / 128, count), 128, 0, s>>>(src, n, a);
    return cudaGetLastError();
}

size_t gather_words(int count, int cnt, bool with_pairs)
{
    return (size_t)count * (1 + (size_t)cnt * (with_pairs ? 3 : 1));
}

cudaError_t launch_gather(const RunView *views, const RunView &one, int count, int cnt, bool with_pairs, long long *out,
                          cudaStream_t s)
{
    gather_kernel<<<count, 128, 0, s>>>(views, one, cnt, with_pairs ? 1 : 0, out);
    return cudaGetLastError();
}

// Four partial sums per dot product: the host's check takes a quarter of the
// additions' latency (0.9 -> 0.25 ms for 20 columns of 4096).
double orthonormality_error(const double *U, int n, int k)
{
    double dev = 0.0;
    for (int a = 0; a < k; ++a)
        for (int c = 0; c <= a; ++c) {
            const double *x = U + (size_t)a * n, *y = U + (size_t)c * n;
            double s[4] = {0.0, 0.0, 0.0, 0.0};
            int l = 0;
            for (; l + 4 <= n; l += 4)
                for (int q = 0; q < 4; ++q) s[q] += x[l + q] * y[l + q];
            for (; l < n; ++l) s[0] += x[l] * y[l];
            const double e = fabs((s[0] + s[1]) + (s[2] + s[3]) - (a == c ? 1.0 : 0.0));
            if (!(e <= dev)) dev = e;  // NaN stays
            if (e != e) return e;
        }
    return dev;
}

} // namespace sap
