// Estimator: block iterative hard thresholding, one small CTA per token (the iteration itself is
// recover_core.cuh), plus the support-drift count.
#include "sense.cuh"

namespace cs {

// M = I - mu Phi^T Phi, row-major with padded rows; only Phi and mu enter, so it can be formed beside the sketch.
__global__ void __launch_bounds__(kGramThreads) gram_kernel(const float *__restrict__ Phi, float mu, int m, int G,
                                                            float *__restrict__ gram) {
    pdl_launch_dependents();
    gram_rows(Phi, mu, m, G, blockIdx.x, gram);
}

// NW = warps = ceil(G / 32).  KC = ceil(k / 8) for k <= 64 (list form), 0 otherwise (dense form).
// DECODE: the form of RecoverOptions::decode (dense).
template <int NW, int KC, bool DECODE>
__global__ void __launch_bounds__(32 * NW) recover_kernel(const __grid_constant__ RecoverArgs a) {
    __shared__ RecoverSmem<NW, KC> s;
    const int g = threadIdx.x;
    pdl_launch_dependents();
    // Phi is a parameter: this thread's column is requested before the wait for the kernel that
    // produces y and M, when it fits 32 registers
    float phc[32];
    if (a.m <= 32) recover_load_phi<NW>(a.Phi, a.m, a.G, g, phc);
    pdl_wait();   // y and M come from the kernel before
    const int t = blockIdx.x;
    recover_row<NW, KC, 0>(
        s, a, GramSource{a.gram, 32 * NW},
        [&](auto &sm) {
            if constexpr (DECODE) y_from_parts<NW, 0>(sm, a.parts, g, t, a.m);
            else for (int i = g; i < a.m; i += 32 * NW) sm.y[i] = ld_dep(a.y + (size_t)t * a.m + i);
        },
        DECODE ? a.mask : nullptr, g, t, phc);
}

typedef void (*RecoverFn)(RecoverArgs);
// k <= G <= 32 NW: the lists a width can meet, and from 65 groups on the dense form.
template <int NW> static RecoverFn recover_fn_kc(int k) {
    const int kc = recover_kc(k);
#define CS_RECOVER(KC) if (kc == KC) return recover_kernel<NW, KC, false>
    CS_RECOVER(1); CS_RECOVER(2); CS_RECOVER(3); CS_RECOVER(4);
    if constexpr (NW > 1) { CS_RECOVER(5); CS_RECOVER(6); CS_RECOVER(7); CS_RECOVER(8); }
#undef CS_RECOVER
    if constexpr (NW > 2) return recover_kernel<NW, 0, false>;
    return nullptr;
}
static RecoverFn recover_fn(int G, int k) {
    switch ((G + 31) / 32) {
        case 1: return recover_fn_kc<1>(k);
        case 2: return recover_fn_kc<2>(k);
        case 3: return recover_fn_kc<3>(k);
        default: return recover_fn_kc<4>(k);
    }
}
// In front of the decode GEMMs, which take over up to 64 groups per token: the dense form, 65 groups at least.
static RecoverFn recover_decode_fn(int G) { return G <= 96 ? recover_kernel<3, 0, true> : recover_kernel<4, 0, true>; }
RecoverArgs recover_args(const cs_plan *plan, const float *Phi, float mu, const float *y, int B, int32_t *support, float *z,
                         float *resid, const RecoverOptions &o) {
    const cs_config &c = plan->cfg;
    RecoverArgs a{};
    a.Phi = Phi; a.gram = plan->gram; a.y = y; a.mu = mu; a.tgamma = 2.f * mu * o.gamma;
    a.m = c.m; a.G = plan->G; a.k = c.k; a.T = o.T < 0 ? c.T : o.T; a.B = B;
    a.support = support; a.z = z; a.resid = resid;
    a.sup0 = o.sup0; a.z0 = o.z0; a.sup_prev = o.sup_prev; a.z_prev = o.z_prev;
    a.check = o.check; a.delta = o.delta; a.drift = o.drift;
    if (o.decode) {
        a.mask = plan->mask; a.mask_count = plan->mask_count;
        a.parts = SketchParts{sketch_partials(plan), o.norm ? sketch_square_partials(plan, B) : nullptr, c.d / 64, B, c.d, c.rms_eps,
                              plan->y_buf};
    }
    a.status = plan->status;
    return a;
}

static SenseFn sense_fn(int G, int k, SenseKind kind, bool all) {
    switch ((G + 31) / 32) {
        case 1: return sense_fn_kc<1>(k, kind, all);
        case 2: return sense_fn_kc<2>(k, kind, all);
        case 3: return sense_fn_kc<3>(k, kind, all);
        default: return sense_fn_kc<4>(k, kind, all);
    }
}

cs_status launch_sense_recover(cs_plan *plan, const float *S, const float *Phi, float mu, const float *x, const float *gamma, int B,
                               float *n_out, int32_t *support, float *z, float *resid, cudaStream_t st, const RecoverOptions &o, int blocks,
                               int n) {
    const cs_config &c = plan->cfg;
    const int pitch = (plan->G + 3) & ~3, row_bytes = c.d / kSenseCtas * 4;
    const int fixed = (plan->G * pitch + c.m * (pitch + 4)) * 4;
    SenseArgs sa{S, x, gamma, c.rms_eps, c.d, min(c.m, (kSenseSmem - fixed) / row_bytes - 1), plan->y_buf, n_out, blocks, 1.f / (float)n};
    {
        StageTimer timer(plan, CS_STAGE_SKETCH, st);
        plan->stage_seen[CS_STAGE_RECOVER] = 0;   // part of this launch
        const bool plain = o.sup0 == nullptr && o.gamma == 0.f && o.check == nullptr && o.delta == nullptr && o.drift == nullptr;
        const SenseKind kind = blocks > 0 ? kSenseStaged : !plain ? kSenseOptions : gamma != nullptr ? kSensePlainNorm : kSensePlain;
        launch_pdl(true, sense_fn(plan->G, c.k, kind, sa.s_rows == c.m), dim3(kSenseCtas * B), dim3(kSenseThreads), (size_t)fixed + (size_t)(sa.s_rows + (blocks > 0)) * row_bytes, st,
                   sa, recover_args(plan, Phi, mu, nullptr, B, support, z, resid, o));
    }
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

// Up to how many tokens the sensing launch takes over from the sketch and recovery launches: as many clusters as the device
// holds at once (15 of eight CTAs on B200; the sixteenth costs 2.5 us of a 15 us step).  None where a CTA's part of S is
// above 128 KB, which the cluster reads anew for every token and the sketch launch once for all of them (d = 5120, m = 64, 2 tokens
// 31.4 us against 28.8; at 8192 x 32 still 23.2 against 23.8 for one token, 34.0 against 32.7 for two), nor for the dense
// form, whose rows of M every thread first reads from shared memory (128 groups, k = 64 in the dense form, one token 52.9 against 47.0).
// Below that it saves 0.5 to 1.5 us a step up to three tokens and is even, within 0.5 us, above.
static int sense_tokens(const cs_plan *plan, int smem) {
    const cs_config &c = plan->cfg;
    if ((size_t)c.m * c.d * 4 > (size_t)kSenseCtas * 128 * 1024 || recover_kc(c.k) == 0) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kSenseCtas * kSenseMaxTokens); cfg.blockDim = dim3(kSenseThreads); cfg.dynamicSmemBytes = smem;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, sense_fn(plan->G, c.k, kSensePlain, true), &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    return min(clusters, kSenseMaxTokens);
}

cs_status prepare_recover(cs_plan *plan) {
    for (SenseKind kind : {kSensePlain, kSensePlainNorm, kSenseOptions, kSenseStaged})
        for (bool all : {false, true})
            CS_CUDA_TRY(plan, cudaFuncSetAttribute(sense_fn(plan->G, plan->cfg.k, kind, all), cudaFuncAttributeMaxDynamicSharedMemorySize, kSenseSmem));
    plan->sense_tokens = sense_tokens(plan, kSenseSmem);
    if (!decode_recovers(plan)) CS_CUDA_TRY(plan, prefer_shared(recover_decode_fn(plan->G)));
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
    launch_pdl(true, o.decode ? recover_decode_fn(G) : recover_fn(G, c.k), dim3(B), dim3(gram_pitch(G)), 0, st,
               recover_args(plan, Phi, mu, y, B, support, z, resid, o));
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

constexpr int kDriftThreads = kMaxG;
__global__ void __launch_bounds__(kDriftThreads)
support_drift_kernel(const int32_t *__restrict__ prev, const int32_t *__restrict__ cur, int k,
                     int32_t *__restrict__ drift, float *__restrict__ ratio) {
    const int t = blockIdx.x;
    drift_row<0, kDriftThreads>(prev + (size_t)t * k, cur + (size_t)t * k, k, threadIdx.x, t, drift, ratio);
}

cs_status launch_support_drift(cs_plan *plan, const int32_t *prev, const int32_t *cur, int B, int32_t *drift,
                               float *ratio, cudaStream_t st) {
    support_drift_kernel<<<B, kDriftThreads, 0, st>>>(prev, cur, plan->cfg.k, drift, ratio);
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

}  // namespace cs
