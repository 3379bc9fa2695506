// basis_forms.cuh -- a new basis in every form the kernels read, and the
// results of runs gathered for one copy (basis_forms.cu).
#pragma once

#include "sap_internal.cuh"

namespace sap {

constexpr int kMaxForms = 20;  // bases of one upload (a dimension sweep's)

struct BasisForms {
    double *U64;          // n x k column-major
    float *U32, *U32lo;   // n x KP row-major, pad columns zero
    void *Uhi, *Ulo;      // k rows of NP 16-bit operands, or null (FP64 data)
    ProbState *st;        // reset to the state before the first evaluation (null: left alone)
    int k, KP, NP;
};
struct BasisFormsArgs {
    BasisForms b[kMaxForms];
    int bf16;             // operand split
    int hist_cap;
};
// Basis q takes the first k columns of src (device, n rows, column-major).
cudaError_t launch_basis_forms(const double *src, int n, const BasisFormsArgs &a, int count, cudaStream_t s);

struct RunView {
    const double *hist;
    const int2 *am;
    ProbState *st;
};
// 64-bit words launch_gather writes: the status words (cleared on the
// device), then the ratios, then the pairs (two words each).
size_t gather_words(int count, int cnt, bool with_pairs);
cudaError_t launch_gather(const RunView *views, const RunView &one, int count, int cnt, bool with_pairs, long long *out,
                          cudaStream_t s);

// max |U^T U - I| of an n x k column-major basis (host); NaN if any entry is.
double orthonormality_error(const double *U, int n, int k);

} // namespace sap
