// Estimator: block iterative hard thresholding, one small CTA per token (the iteration itself is
// recover_core.cuh), plus the support-drift count.
#include "recover_core.cuh"

namespace cs {

// M = I - mu Phi^T Phi, row-major with padded rows; only Phi and mu enter, so it can be formed beside the sketch.
__global__ void __launch_bounds__(kGramThreads) gram_kernel(const float *__restrict__ Phi, float mu, int m, int G,
                                                            float *__restrict__ gram) {
    pdl_launch_dependents();
    gram_rows(Phi, mu, m, G, blockIdx.x, gram);
}

// Support drift between consecutive decoding steps (Sec. 11): Delta_t = |S_t symmetric-difference
// S_{t-1}|.  Both rows are ascending and distinct, so entry j of the new row is looked up in the old
// one by bisection; the rows have k entries each, so the symmetric difference is twice the misses.
// Called by a whole CTA of at least k threads.
__device__ __forceinline__ void drift_row(const int32_t *p, const int32_t *cur, int k, int j, int t, int32_t *drift, float *ratio) {
    int missing = 0;
    if (j < k) {
        const int e = ld_dep(cur + j);
        int lo = 0, hi = k;                       // first index whose entry is >= e
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (ld_dep(p + mid) < e) lo = mid + 1; else hi = mid;
        }
        missing = !(lo < k && ld_dep(p + lo) == e);
    }
    const int n = __syncthreads_count(missing);
    if (j == 0) {
        if (drift != nullptr) drift[t] = 2 * n;
        // D_t = |S_t sym.diff S_{t-1}| / |S_t union S_{t-1}| (Sec. 15): both rows have k entries, so the union has k + n
        if (ratio != nullptr) ratio[t] = (float)(2 * n) / (float)(k + n);
    }
}

// The previous supports of a recovery: validated (ascending, distinct, in range), and the drift against them.
struct RecoverDrift {
    const int32_t *prev;
    int32_t *delta;
    float *ratio;
};

// The sketch of a token as launch_sketch_slices leaves it: partial sums per slice of columns.
struct SketchParts {
    const float *y, *ss;       // [slices][B, m] and, with an RMSNorm, [slices][B]; y == NULL: the sketch is given
    int slices, B, d;
    float eps;
    float *y_out, *rscale;     // [B, m], [B]
};

// s.y of token t from the partials: thread g adds the slices of one row in its share of the slices, the shares are added
// in order; the row scale is folded in.
template <int NW, typename Smem>
__device__ __forceinline__ void y_from_parts(Smem &s, const SketchParts &p, int g, int t, int m) {
    constexpr int GP = 32 * NW;
    const int shares = GP / m < 1 ? 1 : GP / m;            // threads per row (m <= 64 <= 2 GP)
    for (int row0 = 0; row0 < m; row0 += GP) {             // one round unless m > GP
        const int row = row0 + g % m, share = g / m;
        float a = 0.f;
        if (row < m && share < shares) {
            const int n = (p.slices + shares - 1) / shares, lo = share * n, hi = min(p.slices, lo + n);
            const float *src = p.y + (size_t)t * m + row;
            for (int i = lo; i < hi; i += 16) {
                float v[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) v[u] = i + u < hi ? ld_dep(src + (size_t)(i + u) * p.B * m) : 0.f;
#pragma unroll
                for (int u = 0; u < 16; ++u) a += v[u];
            }
        }
        if (m > GP) { if (row < m) s.y[row] = a; }
        else s.part[g] = a;
    }
    float rs = 1.f;
    if (p.ss != nullptr) {   // every warp for itself
        float q = 0.f;
        for (int i = g & 31; i < p.slices; i += 32) q += ld_dep(p.ss + (size_t)i * p.B + t);
        rs = rsqrtf(warp_sum(q) / (float)p.d + p.eps);
        if (g == 0) p.rscale[t] = rs;
    }
    bar_sync<0, GP>();
    for (int row = g; row < m; row += GP) {
        float a = 0.f;
        if (m > GP) a = s.y[row];
        else for (int sh = 0; sh < shares; ++sh) a += s.part[sh * m + row];
        a *= rs;
        s.y[row] = a;
        p.y_out[(size_t)t * m + row] = a;
    }
}

// NW = warps = ceil(G / 32).  KC = ceil(k / 8) for k <= 56 (list form), 0 otherwise (dense form).
// DECODE: the form of RecoverOptions::decode.
template <int NW, int KC, bool DECODE>
__global__ void __launch_bounds__(32 * NW)
recover_kernel(const float *__restrict__ Phi, const float *__restrict__ gram, float mu, const float *__restrict__ y,
               int m, int G, int k, int T, int32_t *__restrict__ support, float *__restrict__ z_out,
               float *__restrict__ resid_out, const int32_t *__restrict__ sup0, const float *__restrict__ z0,
               float tgamma, const int32_t *__restrict__ sup_prev, const float *__restrict__ z_prev, uint32_t *__restrict__ mask,
               SketchParts parts, RecoverDrift drift, DeviceStatus *status) {
    __shared__ RecoverSmem<NW, KC> s;
    const int g = threadIdx.x, t = blockIdx.x;
    if (!DECODE) pdl_launch_dependents();
    // Phi is a parameter: this thread's column is requested before the wait for the kernel that
    // produces y and M, when it fits 32 registers
    float phc[32];
    if (m <= 32) recover_load_phi<NW>(Phi, m, G, g, phc);
    pdl_wait();   // y and M come from the kernel before
    // The decode GEMMs read what the kernels before this one wrote without a wait of their own, and wait for the
    // supports behind their main loop.
    if (DECODE) pdl_launch_dependents();
    if (drift.prev != nullptr && g < k) {
        const int32_t *p = drift.prev + (size_t)t * k + g;
        const int e = ld_dep(p);
        if (e < 0 || e >= G || (g > 0 && ld_dep(p - 1) >= e)) atomicCAS(&status->code, 0, (int)CS_ERR_SUPPORT);
    }
    recover_token<NW, KC, 0>(s, g, Phi, GramSource{gram, 32 * NW}, mu,
                             [&](auto &sm) {
                                 if constexpr (DECODE) y_from_parts<NW>(sm, parts, g, t, m);
                                 else for (int row = g; row < m; row += 32 * NW) sm.y[row] = ld_dep(y + (size_t)t * m + row);
                             }, m, G, k, T, support + (size_t)t * k,
                             z_out != nullptr ? z_out + (size_t)t * k : nullptr,
                             resid_out != nullptr ? resid_out + t : nullptr,
                             sup0 != nullptr ? sup0 + (size_t)t * k : nullptr, z0 != nullptr ? z0 + (size_t)t * k : nullptr,
                             tgamma, sup_prev != nullptr ? sup_prev + (size_t)t * k : nullptr,
                             z_prev != nullptr ? z_prev + (size_t)t * k : nullptr,
                             DECODE ? mask + (size_t)t * 4 : nullptr, status, phc, [] {}, [](int, int) {}, [] {});
    if (drift.delta != nullptr || drift.ratio != nullptr) {
        __syncthreads();   // the support row is written
        drift_row(drift.prev + (size_t)t * k, support + (size_t)t * k, k, g, t, drift.delta, drift.ratio);
    }
}

typedef void (*RecoverFn)(const float *, const float *, float, const float *, int, int, int, int, int32_t *, float *, float *,
                          const int32_t *, const float *, float, const int32_t *, const float *, uint32_t *, SketchParts, RecoverDrift, DeviceStatus *);
static int recover_kc(int k) { return k <= 56 ? (k + 7) / 8 : 0; }
template <int NW, bool DECODE> static RecoverFn recover_fn_kc(int k) {
    switch (recover_kc(k)) {
        case 1: return recover_kernel<NW, 1, DECODE>;
        case 2: return recover_kernel<NW, 2, DECODE>;
        case 3: return recover_kernel<NW, 3, DECODE>;
        case 4: return recover_kernel<NW, 4, DECODE>;
        case 5: return recover_kernel<NW, 5, DECODE>;
        case 6: return recover_kernel<NW, 6, DECODE>;
        case 7: return recover_kernel<NW, 7, DECODE>;
        default: return recover_kernel<NW, 0, DECODE>;
    }
}
template <bool DECODE> static RecoverFn recover_fn(int G, int k) {
    switch ((G + 31) / 32) {
        case 1: return recover_fn_kc<1, DECODE>(k);
        case 2: return recover_fn_kc<2, DECODE>(k);
        case 3: return recover_fn_kc<3, DECODE>(k);
        default: return recover_fn_kc<4, DECODE>(k);
    }
}
cs_status prepare_recover(cs_plan *plan) {
    CS_CUDA_TRY(plan, prefer_shared(recover_fn<true>(plan->G, plan->cfg.k)));
    return CS_OK;
}

cs_status launch_recover(cs_plan *plan, const float *Phi, float mu, const float *y, int B, int32_t *support,
                         float *z, float *resid, bool gram_ready, cudaStream_t st, const RecoverOptions &o) {
    const cs_config &c = plan->cfg;
    const int G = plan->G;
    StageTimer timer(plan, CS_STAGE_RECOVER, st);
    if (!gram_ready) {
        launch_pdl(true, gram_kernel, dim3(gram_blocks(G)), dim3(kGramThreads), 0, st, Phi, mu, c.m, G, plan->gram);
        plan->launches++;
        CS_CUDA_TRY(plan, cudaGetLastError());
    }
    SketchParts parts{};
    if (o.decode)
        parts = SketchParts{sketch_partials(plan), o.norm ? sketch_square_partials(plan, B) : nullptr, c.d / 64, B, c.d, c.rms_eps,
                            plan->y_buf, plan->rscale};
    launch_pdl(true, o.decode ? recover_fn<true>(G, c.k) : recover_fn<false>(G, c.k), dim3(B), dim3(gram_pitch(G)), 0, st, Phi, (const float *)plan->gram, mu, y, c.m, G, c.k,
               o.T < 0 ? c.T : o.T, support, z, resid, o.sup0, o.z0, 2.f * mu * o.gamma, o.sup_prev, o.z_prev,
               o.decode ? plan->mask : (uint32_t *)nullptr, parts, RecoverDrift{o.check, o.delta, o.drift}, plan->status);
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

constexpr int kDriftThreads = kMaxG;
__global__ void __launch_bounds__(kDriftThreads)
support_drift_kernel(const int32_t *__restrict__ prev, const int32_t *__restrict__ cur, int k,
                     int32_t *__restrict__ drift, float *__restrict__ ratio) {
    const int t = blockIdx.x;
    drift_row(prev + (size_t)t * k, cur + (size_t)t * k, k, threadIdx.x, t, drift, ratio);
}

cs_status launch_support_drift(cs_plan *plan, const int32_t *prev, const int32_t *cur, int B, int32_t *drift,
                               float *ratio, cudaStream_t st) {
    support_drift_kernel<<<B, kDriftThreads, 0, st>>>(prev, cur, plan->cfg.k, drift, ratio);
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

}  // namespace cs
