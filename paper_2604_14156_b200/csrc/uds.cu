// Uncertainty-driven sensing controller (Sec. 8.1): the predictive entropy of the previous step's
// distribution over the vocabulary, H = -sum_v p_v log p_v with p = softmax(logits), and the
// measurement budget it sets, m = clip(floor(m_base (1 + gamma H)), m_min, m_max).
//
// One pass over the logits, one launch.  Every thread keeps the three moments of its elements
//     M = max l,   Z = sum e^(l - M),   W = sum e^(l - M) (l - M);
// a row is split over a cluster of up to eight CTAs.  Moments are folded by taking the common maximum first, one rescale per
// thread, then plain sums in a fixed order (warp, CTA, cluster over distributed shared memory); CTA 0 ends with
//     H = log Z - W / Z.
// Small batches are a latency chain (at 11 tokens of 32000 logits one load round trip and the folds): as two launches, the row's
// moments merged pairwise with two exponentials a merge and folded by the second launch, 1 x 32000 logits took 5.6 us and 11 x 32000 5.7,
// now 2.6 and 2.8.  Large ones are bound by HBM and the arithmetic: 64 x 128256 16.6 and 10.9 us, 512 x 128256 66.6 and 52.9 (5.0 TB/s).
#include "cs_internal.cuh"

namespace cs {

constexpr int kUdsThreads = 512;
constexpr int kUdsWarps = kUdsThreads / 32;
constexpr int kUdsMaxCtas = 8;   // of a cluster

struct Moments { float M, Z, W; };   // Z == 0: no element yet

// Folds a batch of N elements: one rescale to the batch maximum, then N independent exponentials.
// Entries of -inf contribute nothing (p = 0, 0 log 0 = 0).
template <int N>
__device__ __forceinline__ void add_logits(Moments &s, const float (&v)[N]) {
    float m = v[0];
#pragma unroll
    for (int j = 1; j < N; ++j) m = fmaxf(m, v[j]);
    if (m == -INFINITY) {                         // nothing but -inf, or a NaN among it (fmaxf passes a NaN over)
        bool nan = false;
#pragma unroll
        for (int j = 0; j < N; ++j) nan |= v[j] != v[j];
        if (nan) s.Z = NAN;                       // (stays one in every fold below)
        return;
    }
    if (s.Z == 0.f) {
        s.M = m;
    } else if (m > s.M) {                         // new maximum: rescale what has been summed
        const float dm = s.M - m, sc = expf(dm);
        s.W = sc > 0.f ? sc * (s.W + dm * s.Z) : 0.f;
        s.Z = sc * s.Z;
        s.M = m;
    }
    float z0 = 0.f, z1 = 0.f, w0 = 0.f, w1 = 0.f;
#pragma unroll
    for (int j = 0; j < N; j += 2) {
        const float d0 = v[j] - s.M, d1 = v[j + 1] - s.M;
        const float e0 = __expf(d0), e1 = __expf(d1);   // d <= 0: the fast exponential's error (about
                                                        // 1e-7 |d| relative) is far inside the 1e-5 asked of H
        z0 += e0; z1 += e1;
        w0 += e0 > 0.f ? e0 * d0 : 0.f;           // e = 0 (underflow, or a -inf entry): no term
        w1 += e1 > 0.f ? e1 * d1 : 0.f;
    }
    s.Z += z0 + z1;
    s.W += w0 + w1;
}

// The same moments about a maximum M (>= s.M where s has an element; a NaN of either stays one).
__device__ __forceinline__ void rescale(Moments &s, float M) {
    if (s.Z == 0.f) { s.M = M; return; }
    const float dm = s.M - M, sc = expf(dm);
    s.W = sc > 0.f || sc != sc ? sc * (s.W + dm * s.Z) : 0.f;
    s.Z = sc * s.Z;
    s.M = M;
}
// Folds the moments of a warp's lanes: every lane ends with the same bits.
__device__ __forceinline__ void warp_fold(Moments &s) {
    float M = s.Z == 0.f ? -INFINITY : s.M;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    rescale(s, M);
    s.Z = warp_sum(s.Z);
    s.W = warp_sum(s.W);
}

// grid: B rows of `ctas` CTAs, which are one cluster: CTA s of row t takes elements [s * per, min(V, (s + 1) * per)), N of a
// thread in flight.  The floor is taken in double precision from the f32 entropy; a NaN entropy (a NaN or +inf logit) asks for m_max.
template <int N>
__global__ void __launch_bounds__(kUdsThreads)
uds_kernel(const float *__restrict__ logits, int V, int ctas, int per, float m_base, float gamma, int m_min, int m_max, float *__restrict__ H_out,
           int32_t *__restrict__ m_out) {
    __shared__ Moments warp_s[kUdsWarps], cta_s[kUdsMaxCtas];
    const int t = blockIdx.x / ctas, s = blockIdx.x - t * ctas, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lo = s * per, hi = min(V, lo + per);
    const float *row = logits + (size_t)t * V;
    Moments acc{0.f, 0.f, 0.f};
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");   // CTA 0 has started, see below
    pdl_wait();   // the logits may come from the kernel before
    // Not earlier: the launch behind reads its parameters (S, Phi, weights) before its own wait, and what was enqueued ahead of this
    // call may have written them.  From here on that has completed.
    pdl_launch_dependents();
    int i = lo + (int)threadIdx.x;
    for (int end = lo + N * kUdsThreads; end < hi; end += N * kUdsThreads, i += N * kUdsThreads) {   // whole batches
        float v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) v[j] = ld_dep(row + i + j * kUdsThreads);
        add_logits(acc, v);
    }
    if (i < hi) {
        float v[N];
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const int idx = i + j * kUdsThreads;
            v[j] = ld_dep(row + min(idx, hi - 1));
            if (idx >= hi) v[j] = -INFINITY;
        }
        add_logits(acc, v);
    }
    warp_fold(acc);
    if (lane == 0) warp_s[warp] = acc;
    __syncthreads();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 0) {
        acc = lane < kUdsWarps ? warp_s[lane] : Moments{0.f, 0.f, 0.f};
        warp_fold(acc);
        if (lane == 0) {
            uint32_t dst;
            asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst) : "r"((uint32_t)__cvta_generic_to_shared(&cta_s[s])));
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(acc.M) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 4u), "f"(acc.Z) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 8u), "f"(acc.W) : "memory");
        }
        __syncwarp();
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (s != 0 || warp != 0) return;
    acc = lane < ctas ? cta_s[lane] : Moments{0.f, 0.f, 0.f};
    warp_fold(acc);
    if (lane == 0) {
        float H = acc.Z > 0.f ? fmaxf(logf(acc.Z) - acc.W / acc.Z, 0.f) : (acc.Z == 0.f ? 0.f : acc.Z);
        if (acc.Z != acc.Z || acc.W != acc.W) H = NAN;
        int m = m_max;
        if (H == H) {
            const double x = floor((double)m_base * (1.0 + (double)gamma * (double)H));
            m = x >= (double)m_max ? m_max : (x <= (double)m_min ? m_min : (int)x);
        }
        if (H_out != nullptr) H_out[t] = H;
        m_out[t] = m;
    }
}

cs_status launch_uds_budget(cs_plan *plan, const float *logits, int B, int V, float m_base, float gamma,
                            int m_min, int m_max, float *H, int32_t *m_t, cudaStream_t st) {
    // about two CTAs per SM, each with 2048 elements at least
    int ctas = 1;
    while (ctas < kUdsMaxCtas && 2 * ctas * B <= 2 * plan->sm_count && V >= 2 * ctas * 2048) ctas *= 2;
    const int per = (V + ctas - 1) / ctas;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas * B); cfg.blockDim = dim3(kUdsThreads); cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = ctas; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    // 16 logits of a thread in flight where the CTAs are too few to keep the memory busy with 8
    const bool deep = per > 8 * kUdsThreads && ctas * B <= 2 * plan->sm_count;
    cudaLaunchKernelEx(&cfg, deep ? uds_kernel<16> : uds_kernel<8>, logits, V, ctas, per, m_base, gamma, m_min, m_max, H, m_t);
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

}  // namespace cs
