// colmean.cuh -- column means of an N x n row-major matrix in FP64, shared by
// the length preparation (restructured.cu) and the PCA start (pca.cu).
//
// One thread per column walked all N rows in sequence (824 us at N = 8000, n
// = 90: one load latency per row).  The rows are cut into bands instead: a
// block sums 32 columns of one band (8 threads per column), a second launch
// adds the bands in order.  The summation order is fixed, so the means are
// reproducible; 8 us at that size, bound by the two launches.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>

namespace sap {

constexpr int kMeanBands = 64;

inline int colmean_bands(int N) { return std::min(kMeanBands, (N + 127) / 128); }
inline size_t colmean_scratch(int N, int n) { return (size_t)colmean_bands(N) * n; }

template <typename TX>
__global__ void __launch_bounds__(256) colsum_kernel(const TX *X, int N, int n, int rows, double *part)
{
    __shared__ double sh[8][33];
    const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int l = blockIdx.x * 32 + c, r0 = blockIdx.y * rows, r1 = min(N, r0 + rows);
    double acc = 0.0;
    if (l < n)
#pragma unroll 8
        for (int i = r0 + g; i < r1; i += 8) acc += (double)X[(size_t)i * n + l];
    sh[g][c] = acc;
    __syncthreads();
    if (g == 0 && l < n) {
        for (int q = 1; q < 8; ++q) acc += sh[q][c];
        part[(size_t)blockIdx.y * n + l] = acc;
    }
}

template <typename TM>
__global__ void __launch_bounds__(128) colmean_kernel(const double *part, int bands, int N, int n, TM *mean)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n) return;
    double acc = 0.0;
#pragma unroll 4
    for (int b = 0; b < bands; ++b) acc += part[(size_t)b * n + l];
    mean[l] = (TM)(acc / N);
}

// mean: n entries; part: colmean_scratch(N, n) doubles of scratch.
template <typename TX, typename TM>
cudaError_t launch_colmean(const TX *X, int N, int n, double *part, TM *mean, cudaStream_t s)
{
    const int bands = colmean_bands(N), rows = (N + bands - 1) / bands;
    colsum_kernel<TX><<<dim3((n + 31) / 32, bands), 256, 0, s>>>(X, N, n, rows, part);
    colmean_kernel<TM><<<(n + 127) / 128, 128, 0, s>>>(part, bands, N, n, mean);
    return cudaGetLastError();
}

} // namespace sap
