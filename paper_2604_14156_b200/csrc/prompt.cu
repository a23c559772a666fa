// Prompt-level support: the column sums behind the mean hidden state of the prompt (the mean sketch is S applied to it,
// and the sensing launch folds the row blocks and divides).
//
// colsum[b, i] = sum over the rows of block b of H[t, i], H [n, d] bf16.  A CTA takes 256 columns (eight per thread,
// 16-byte loads, eight in flight) and the rows of one block, dealt to eight warps that are added in order.  Bound by
// HBM: 7.4 us for the 21 MB of 2048 tokens at d = 5120, 11.4 us for 4096 (with 4-byte loads 9.5 and 15 us, and the fold
// was a launch of its own, 4.6 us; with a branch around each load instead of a clamped row 11.6 us).
#include "cs_internal.cuh"

namespace cs {

constexpr int kMeanThreads = 256;
constexpr int kMeanWarps = kMeanThreads / 32;

__device__ __forceinline__ uint4 ld_cg(const void *p) {   // from L2: the producer may have finished after this CTA began
    uint4 r;
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p) : "memory");
    return r;
}

__global__ void __launch_bounds__(kMeanThreads)
colsum_kernel(const __nv_bfloat16 *__restrict__ H, int n, int d, int rows_per_block, float *__restrict__ colsum) {
    __shared__ float part[kMeanWarps][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int col = blockIdx.x * 256 + lane * 8;
    const int r0 = blockIdx.y * rows_per_block, r1 = min(n, r0 + rows_per_block);
    pdl_launch_dependents();
    pdl_wait();   // H may be the previous kernel's output
    float s[8] = {};
    if (col < d) {   // d is a multiple of 64
        for (int r = r0 + warp; r < r1; r += 8 * kMeanWarps) {
            uint4 q[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) q[u] = ld_cg(H + (size_t)min(r + u * kMeanWarps, r1 - 1) * d + col);
#pragma unroll
            for (int u = 1; u < 8; ++u)
                if (r + u * kMeanWarps >= r1) q[u] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                float f[8];
                Chunk<__nv_bfloat16>::widen(q[u], f);
#pragma unroll
                for (int e = 0; e < 8; ++e) s[e] += f[e];
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 8; e += 4) *reinterpret_cast<float4 *>(&part[warp][lane * 8 + e]) = make_float4(s[e], s[e + 1], s[e + 2], s[e + 3]);
    __syncthreads();
    const int c = blockIdx.x * 256 + threadIdx.x;
    if (c < d) {
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kMeanWarps; ++w) t += part[w][threadIdx.x];
        colsum[(size_t)blockIdx.y * d + c] = t;
    }
}

cs_status prepare_prompt(cs_plan *plan) {
    CS_CUDA_TRY(plan, prefer_shared(colsum_kernel));   // the sensing launch's 220 KB start beside it
    return CS_OK;
}

cs_status launch_prompt_colsum(cs_plan *plan, const void *H, int n, int *blocks, cudaStream_t st) {
    const int d = plan->cfg.d;
    const int rpb = (n + min(kMeanRowBlocks, n) - 1) / min(kMeanRowBlocks, n);
    *blocks = (n + rpb - 1) / rpb;
    launch_pdl(true, colsum_kernel, dim3((d + 255) / 256, *blocks), dim3(kMeanThreads), 0, st, static_cast<const __nv_bfloat16 *>(H), n, d,
               rpb, plan->colsum);
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

}  // namespace cs
