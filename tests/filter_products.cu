// The contraction of the all-pairs filter for one 128 x 128 tile: operand
// images in, products out.
#include <cuda_runtime.h>
#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

using namespace sap;

__global__ void __launch_bounds__(128) products_kernel(const unsigned char *images, int ksteps, float *out, int *status)
{
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t full, done;
    __shared__ uint32_t slot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t img = ksteps * 4096u;
    const long long budget = 1000000000ll;
    if (tid == 0) {
        tc::mbar_init(&full, 1);
        tc::mbar_init(&done, 1);
        tc::fence_mbar_init();
    }
    if (warp == 0) tc::tmem_alloc(&slot, 128);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tbase = slot;
    if (tid == 0) {
        tc::mbar_expect_tx(&full, 2 * img);
        tc::bulk_g2s(sm, images, 2 * img, &full);
        if (tc::mbar_wait_bounded(&full, 0, budget)) {
            const uint32_t sa = tc::smem_u32(sm), sb = sa + img;
            for (int q = 0; q < ksteps; ++q)
                tc::mma_f16(tbase, tc::desc_k_plain(sa + q * 4096, 2048, 128), tc::desc_k_plain(sb + q * 4096, 2048, 128),
                            tc::idesc_f16(128, 128, 0), q > 0 ? 1u : 0u);
            tc::mma_commit(&done);
        } else {
            *status = 1;
        }
    }
    __syncwarp();
    if (__all_sync(0xffffffffu, tc::mbar_wait_bounded(&done, 0, 2 * budget))) {
        tc::tc_fence_after();
        for (int c = 0; c < 128; c += 32) {
            float v[32];
            tc::tmem_ld32(tbase + ((uint32_t)(32 * warp) << 16) + c, v);
            for (int e = 0; e < 32; ++e) out[(32 * warp + lane) * 128 + c + e] = v[e];
        }
    } else if (lane == 0) {
        *status = 1;
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tbase, 128);
    }
}

// images: the A image, then the B image (device memory); out: 128 x 128;
// status: zero on entry, 1 if a wait ran out.  ksteps <= 7.
extern "C" int filter_products(const void *images, int ksteps, float *out, int *status)
{
    if (ksteps < 1 || ksteps > 7) return 1;
    const int bytes = 2 * ksteps * 4096;
    cudaError_t e = cudaFuncSetAttribute(products_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return (int)e;
    products_kernel<<<1, 128, bytes>>>(static_cast<const unsigned char *>(images), ksteps, out, status);
    e = cudaGetLastError();
    return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}
