// The C boundary: plan life cycle, host-side validation and dispatch.  See include/cs.h.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <new>

#include "cs_internal.cuh"

namespace cs {

cs_status record_cuda(cs_plan *plan, cudaError_t e, const char *what) {
    if (plan != nullptr)
        snprintf(plan->cuda_error, sizeof plan->cuda_error, "%s: %s", what, cudaGetErrorString(e));
    return CS_ERR_CUDA;
}

static cs_status check_config(const cs_config *c) {
    if (c->d <= 0 || c->d_ff <= 0 || c->group <= 0 || c->m <= 0 || c->k <= 0 || c->T < 0 || c->max_tokens <= 0)
        return CS_ERR_SHAPE;
    if (c->d_ff % c->group != 0) return CS_ERR_SHAPE;
    const int G = c->d_ff / c->group;
    if (c->k > G) return CS_ERR_SHAPE;
    if (!(c->rms_eps > 0.f) || !isfinite(c->rms_eps)) return CS_ERR_NONFINITE;
    if (c->group != 64 && c->group != 128) return CS_ERR_UNSUPPORTED;
    if (G > kMaxG || c->m > kMaxM || c->d > kMaxD || c->d % 64 != 0) return CS_ERR_UNSUPPORTED;
    if (c->w_dtype != CS_F32 && c->w_dtype != CS_BF16) return CS_ERR_UNSUPPORTED;
    return CS_OK;
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace cs

using namespace cs;

// Device-visible address of page-locked host memory (unified addressing), or NULL for pageable memory.
static void *device_alias(const void *host) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, host) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    return a.type == cudaMemoryTypeHost ? a.devicePointer : nullptr;
}

constexpr size_t kZeroCopyBytes = 64 * 1024;
constexpr size_t kZeroCopyBytesLarge = 4 * 1024 * 1024;

// x (page-locked host memory) -> plan scratch.  Both the load and the store come after the
// programmatic-launch wait: whatever ran before on the stream may have written the host buffer (a
// previous step that stored its result there, when layers are chained through one buffer) and may
// still be reading the scratch copy.
__global__ void __launch_bounds__(256) stage_in_kernel(const float4 *src, float4 *dst, int n4) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    cs::pdl_launch_dependents();
    cs::pdl_wait();
    if (i < n4) {
        float4 v;   // volatile and uncached: the host (or the step before) rewrites the buffer between steps
        asm volatile("ld.volatile.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(src + i) : "memory");
        dst[i] = v;
    }
}

extern "C" {

cs_status cs_plan_create(const cs_config *cfg, cs_plan **out) {
    if (cfg == nullptr || out == nullptr) return CS_ERR_NULL;
    cs_status s = check_config(cfg);
    if (s != CS_OK) return s;
    cs_plan *p = new (std::nothrow) cs_plan();
    if (p == nullptr) return CS_ERR_CUDA;
    memset(p, 0, sizeof *p);
    p->cfg = *cfg;
    p->G = cfg->d_ff / cfg->group;
    cudaError_t e = cudaGetDevice(&p->device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, p->device);
    const size_t nt = (size_t)cfg->max_tokens;
    p->nx_max = max(p->sm_count, (cfg->k * cfg->group + kGatherMaxRows - 1) / kGatherMaxRows);
    auto alloc = [&](void **ptr, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(ptr, bytes);
    };
    alloc((void **)&p->n_buf, nt * cfg->d * sizeof(float));
    alloc((void **)&p->y_buf, nt * cfg->m * sizeof(float));
    alloc((void **)&p->sup_buf, nt * cfg->k * sizeof(int32_t));
    alloc((void **)&p->partial, (size_t)kGatherMaxTokens * p->nx_max * cfg->d * sizeof(float));
    alloc((void **)&p->gram, (size_t)kMaxG * kMaxG * sizeof(float));
    alloc((void **)&p->resid_buf, nt * sizeof(float));
    alloc((void **)&p->fb_flags, nt * sizeof(int32_t));
    alloc((void **)&p->fb_list, nt * sizeof(int32_t));
    alloc((void **)&p->fb_count, sizeof(int32_t));
    alloc((void **)&p->slot_table, nt * kSlotTablePitch * sizeof(int32_t));
    alloc((void **)&p->ticket, nt * sizeof(unsigned));
    alloc((void **)&p->colsum, (size_t)kMeanRowBlocks * cfg->d * sizeof(float));
    alloc((void **)&p->status, sizeof(DeviceStatus));
    p->mma_ok = cfg->w_dtype == CS_BF16 && cfg->group == 128 && cfg->d % 256 == 0;
    // The gather path streams B * k groups, the tensor-core path every group once: it takes over where the first exceeds
    // the second by 15 %.  One step, gather against tensor path, at the last batch on each side of the line: 22 of 86 groups of
    // d = 4096, 4 tokens 44.0 and 48.2 us, 5 tokens 50.5 and 49.6; 9 of 86, 10 tokens 45.1 and 48.8, 11 tokens 46.7 and 47.7, 12
    // 50.7 and 49.5; 12 of 48 of d = 2048, 4 tokens 23.1 and 27.8, 5 tokens 26.5 and 28.7, 6 28.3 and 28.4: there the line is one batch
    // early.  It knows nothing of the row width: at d = 5120, whose rows are 1.25 of the gather's slices, it is late (11 of 108 groups,
    // 8 tokens 71.5 and 65.1, 11 tokens 85.3 and 67.7; 27 of 108, 3 tokens 64.8 both, 4 tokens 79.6 and 66.9); cs_plan_set_crossover moves it.
    p->mma_min_tokens = max(2, min(kMmaMinTokens, (int)ceilf(1.15f * (float)p->G / (float)cfg->k)));
    alloc((void **)&p->mask, nt * 4 * sizeof(uint32_t));
    alloc((void **)&p->mask_count, sizeof(unsigned));
    alloc((void **)&p->counts, (size_t)kMaxG * sizeof(int32_t));
    alloc((void **)&p->offsets, (size_t)(kMaxG + 1) * sizeof(int32_t));
    alloc((void **)&p->token_ids, nt * cfg->k * sizeof(int32_t));
    alloc((void **)&p->glist, (size_t)kMaxG * sizeof(int32_t));
    alloc((void **)&p->nu, sizeof(int32_t));
    if (p->mma_ok) {
        const size_t m_pad = (nt + 127) / 128 * 128;
        p->mma_slices = max(1, min(16, p->sm_count / max(1, cfg->d / 256)));
        alloc((void **)&p->x_bf16, 2 * nt * cfg->d * 2);
        alloc((void **)&p->act, 2 * max(nt, (size_t)128) * cfg->d_ff * 2);
        // slices * padded tokens never exceeds 128 * (SMs / column tiles): see launch_ffn_mma
        const size_t slice_rows = (size_t)128 * (p->sm_count / max(1, cfg->d / 256) + 1);
        const size_t decode_rows = (size_t)decode_slices(p) * min(nt, (size_t)kDecodeMaxTokens);
        alloc((void **)&p->mma_partial, max(max(slice_rows, max(decode_rows, 2 * min(nt, (size_t)kDecodeMaxTokens))), m_pad) * cfg->d * sizeof(float));
    }
    alloc((void **)&p->x_host_in, nt * cfg->d * sizeof(float));
    alloc((void **)&p->x_host_out, nt * cfg->d * sizeof(float));
    for (int i = 0; i < 2 * CS_STAGE_COUNT; ++i)
        if (e == cudaSuccess) e = cudaEventCreate(&p->ev[i]);
    if (e == cudaSuccess) e = cudaMemset(p->status, 0, sizeof(DeviceStatus));
    if (e == cudaSuccess) e = cudaMemset(p->mask_count, 0, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(p->ticket, 0, nt * sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(p->slot_table, 0, nt * kSlotTablePitch * sizeof(int32_t));
    if (e == cudaSuccess && prepare_sketch(p) != CS_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess && prepare_recover(p) != CS_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess && prepare_prompt(p) != CS_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess && prepare_solvers(p) != CS_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess && prepare_ffn_gather(p) != CS_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess && p->mma_ok && prepare_ffn_mma(p) != CS_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess && p->mma_ok && prepare_decode(p) != CS_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess) e = cudaMemset(p->mask, 0, nt * 4 * sizeof(uint32_t));
    if (e != cudaSuccess) {
        cs_plan_destroy(p);
        return CS_ERR_CUDA;
    }
    *out = p;
    return CS_OK;
}

cs_status cs_plan_destroy(cs_plan *p) {
    if (p == nullptr) return CS_ERR_NULL;
    cudaFree(p->n_buf); cudaFree(p->y_buf); cudaFree(p->sup_buf);
    cudaFree(p->partial); cudaFree(p->gram); cudaFree(p->slot_table); cudaFree(p->ticket);
    cudaFree(p->resid_buf); cudaFree(p->fb_flags); cudaFree(p->fb_list); cudaFree(p->fb_count); cudaFree(p->colsum);
    cudaFree(p->status); cudaFree(p->x_host_in); cudaFree(p->x_host_out);
    cudaFree(p->mask); cudaFree(p->mask_count); cudaFree(p->counts); cudaFree(p->offsets); cudaFree(p->token_ids); cudaFree(p->glist);
    cudaFree(p->nu); cudaFree(p->x_bf16); cudaFree(p->act); cudaFree(p->mma_partial);
    for (int i = 0; i < 2 * CS_STAGE_COUNT; ++i)
        if (p->ev[i] != nullptr) cudaEventDestroy(p->ev[i]);
    delete p;
    return CS_OK;
}

cs_status cs_sketch(cs_plan *plan, const float *S, const float *h, int32_t B, float *y, void *stream) {
    if (plan == nullptr || S == nullptr || h == nullptr || y == nullptr) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    if (!aligned16(S) || !aligned16(h)) return CS_ERR_UNSUPPORTED;
    return launch_sketch(plan, S, h, nullptr, B, y, nullptr, nullptr, 0.f, static_cast<cudaStream_t>(stream));
}

cs_status cs_recover(cs_plan *plan, const float *Phi, float mu, const float *y, int32_t B,
                     int32_t *support, float *z, float *resid, void *stream) {
    if (plan == nullptr || Phi == nullptr || y == nullptr || support == nullptr) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    if (!isfinite(mu) || !(mu > 0.f)) return CS_ERR_NONFINITE;
    return launch_recover(plan, Phi, mu, y, B, support, z, resid, false, static_cast<cudaStream_t>(stream));
}

cs_status cs_recover_warm(cs_plan *plan, const float *Phi, float mu, const float *y, int32_t B, int32_t T,
                          const int32_t *support0, const float *z0, int32_t *support, float *z, float *resid,
                          void *stream) {
    if (plan == nullptr || Phi == nullptr || y == nullptr || support0 == nullptr || z0 == nullptr || support == nullptr)
        return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens || T < 1) return CS_ERR_SHAPE;
    if (!isfinite(mu) || !(mu > 0.f)) return CS_ERR_NONFINITE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    RecoverOptions o;
    o.T = T; o.sup0 = support0; o.z0 = z0; o.check = support0;
    return launch_recover(plan, Phi, mu, y, B, support, z, resid, false, st, o);
}

cs_status cs_support_drift(cs_plan *plan, const int32_t *support_prev, const int32_t *support_cur, int32_t B,
                           int32_t *drift, void *stream) {
    if (plan == nullptr || support_prev == nullptr || support_cur == nullptr || drift == nullptr) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cs_status s = launch_check_support(plan, support_prev, B, st);
    if (s == CS_OK) s = launch_check_support(plan, support_cur, B, st);
    if (s != CS_OK) return s;
    return launch_support_drift(plan, support_prev, support_cur, B, drift, nullptr, st);
}

cs_status cs_support_drift_ratio(cs_plan *plan, const int32_t *support_prev, const int32_t *support_cur, int32_t B,
                                 int32_t *delta, float *D, void *stream) {
    if (plan == nullptr || support_prev == nullptr || support_cur == nullptr || (delta == nullptr && D == nullptr))
        return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cs_status s = launch_check_support(plan, support_prev, B, st);
    if (s == CS_OK) s = launch_check_support(plan, support_cur, B, st);
    if (s != CS_OK) return s;
    return launch_support_drift(plan, support_prev, support_cur, B, delta, D, st);
}

static cs_status check_options(const cs_plan *plan, const cs_step_options *o, bool step) {
    if (o->solver != CS_SOLVER_IHT && o->solver != CS_SOLVER_NIHT && o->solver != CS_SOLVER_OMP) return CS_ERR_UNSUPPORTED;
    if (o->solver == CS_SOLVER_OMP && plan->cfg.k > 64) return CS_ERR_UNSUPPORTED;
    if (!isfinite(o->gamma) || o->gamma < 0.f) return CS_ERR_NONFINITE;
    const bool needs_prev = o->warm_start || o->gamma > 0.f;
    if (needs_prev && (o->support_prev == nullptr || o->z_prev == nullptr)) return CS_ERR_NULL;
    if ((o->delta_out != nullptr || o->drift_out != nullptr || (step && o->reuse_support)) && o->support_prev == nullptr)
        return CS_ERR_NULL;
    if ((o->warm_start || o->gamma > 0.f) && o->solver != CS_SOLVER_IHT) return CS_ERR_UNSUPPORTED;
    if (o->warm_start && o->T == 0) return CS_ERR_SHAPE;
    if ((o->srht_sign == nullptr) != (o->srht_rows == nullptr)) return CS_ERR_NULL;
    return CS_OK;
}

// The options of the fixed-step iteration as launch_recover takes them.
static RecoverOptions iht_options(const cs_plan *plan, const cs_step_options *o) {
    RecoverOptions r;
    r.T = o->T < 0 ? plan->cfg.T : o->T; r.gamma = o->gamma;
    if (o->warm_start) { r.sup0 = o->support_prev; r.z0 = o->z_prev; }
    if (o->gamma > 0.f) { r.sup_prev = o->support_prev; r.z_prev = o->z_prev; }
    r.check = o->support_prev;
    r.delta = o->delta_out; r.drift = o->drift_out;
    return r;
}

// The estimator an options struct asks for, on y, with the check of the previous supports and the drift against
// them; gram_ready: plan->gram holds this Phi's matrix.
static cs_status recover_with(cs_plan *plan, const float *Phi, float mu, const float *y, int B, const cs_step_options *o,
                              int32_t *support, float *z, float *resid, bool gram_ready, cudaStream_t st) {
    const int T = o->T < 0 ? plan->cfg.T : o->T;
    if (o->solver == CS_SOLVER_IHT)
        return launch_recover(plan, Phi, mu, y, B, support, z, resid, gram_ready, st, iht_options(plan, o));
    cs_status s = CS_OK;
    if (o->support_prev != nullptr) s = launch_check_support(plan, o->support_prev, B, st);
    if (s == CS_OK)
        s = o->solver == CS_SOLVER_NIHT ? launch_niht(plan, Phi, mu, y, B, T, support, z, resid, st)
                                        : launch_omp(plan, Phi, y, B, support, z, resid, st);
    if (s == CS_OK && (o->delta_out != nullptr || o->drift_out != nullptr))
        s = launch_support_drift(plan, o->support_prev, support, B, o->delta_out, o->drift_out, st);
    return s;
}

cs_status cs_recover_ex(cs_plan *plan, const float *Phi, float mu, const float *y, int32_t B,
                        const cs_step_options *opt, int32_t *support, float *z, float *resid, void *stream) {
    if (opt == nullptr) return cs_recover(plan, Phi, mu, y, B, support, z, resid, stream);
    if (plan == nullptr || Phi == nullptr || y == nullptr || support == nullptr) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    if (!isfinite(mu) || !(mu > 0.f)) return CS_ERR_NONFINITE;
    cs_status s = check_options(plan, opt, false);
    if (s != CS_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return recover_with(plan, Phi, mu, y, B, opt, support, z, resid, false, st);
}

cs_status cs_sketch_srht(cs_plan *plan, const uint32_t *sign_bits, const int32_t *rows, const float *h, int32_t B,
                         float *y, void *stream) {
    if (plan == nullptr || sign_bits == nullptr || rows == nullptr || h == nullptr || y == nullptr) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    return launch_sketch_srht(plan, sign_bits, rows, h, B, y, static_cast<cudaStream_t>(stream));
}

cs_status cs_uds_budget(cs_plan *plan, const float *logits, int32_t B, int32_t V, float m_base, float gamma,
                        int32_t m_min, int32_t m_max, float *H, int32_t *m_t, void *stream) {
    if (plan == nullptr || logits == nullptr || m_t == nullptr) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens || V <= 0 || m_min < 1 || m_max < m_min) return CS_ERR_SHAPE;
    if (!isfinite(m_base) || !(m_base > 0.f) || !isfinite(gamma) || gamma < 0.f) return CS_ERR_NONFINITE;
    return launch_uds_budget(plan, logits, B, V, m_base, gamma, m_min, m_max, H, m_t, static_cast<cudaStream_t>(stream));
}

static cs_status check_weights(const cs_layer *L) {
    if (L == nullptr || L->W_gate == nullptr || L->W_up == nullptr || L->Wd_t == nullptr) return CS_ERR_NULL;
    if (!aligned16(L->W_gate) || !aligned16(L->W_up) || !aligned16(L->Wd_t)) return CS_ERR_UNSUPPORTED;
    return CS_OK;
}

static bool use_decode_mma(const cs_plan *plan, int B) {
    return plan->mma_ok && B >= plan->mma_min_tokens && B <= kDecodeMaxTokens;
}

// Dispatch of the actuator by batch size: gather GEMV, tensor-core decode path, or (more than kDecodeMaxTokens
// tokens) the token-tiled grouped GEMMs over the union list.
// check: the supports come from the caller and are validated on the device (inside the gather
// kernel, or by a small kernel ahead of the tensor-core paths).
static cs_status exec_dispatch(cs_plan *plan, const cs_layer *layer, const float *h, const int32_t *support,
                               int B, const float *residual, float *out, bool check, cudaStream_t st) {
    if (!plan->mma_ok || B < plan->mma_min_tokens)
        return launch_ffn_gather(plan, layer, h, support, B, residual, out, check, st);
    if (use_decode_mma(plan, B)) {
        cs_status s = launch_decode_prep(plan, h, support, B, check, st);
        if (s != CS_OK) return s;
        return launch_decode_ffn(plan, layer, B, nullptr, true, false, residual, out, st);
    }
    if (check) {
        cs_status s = launch_check_support(plan, support, B, st);
        if (s != CS_OK) return s;
    }
    __nv_bfloat16 *x_hi = static_cast<__nv_bfloat16 *>(plan->x_bf16);
    __nv_bfloat16 *x_lo = x_hi + (size_t)plan->cfg.max_tokens * plan->cfg.d;
    cs_status s = launch_split_bf16(plan, h, x_hi, x_lo, (size_t)B * plan->cfg.d, st);
    if (s != CS_OK) return s;
    s = launch_bucket(plan, support, B, st);
    if (s != CS_OK) return s;
    return launch_ffn_mma(plan, layer, x_hi, x_lo, B, plan->glist, plan->nu, 0, plan->mask, residual, out, nullptr, st);
}

cs_status cs_ffn_exec(cs_plan *plan, const cs_layer *layer, const float *h, const int32_t *support,
                      int32_t B, const float *residual, float *out, void *stream) {
    if (plan == nullptr || h == nullptr || support == nullptr || out == nullptr) return CS_ERR_NULL;
    cs_status s = check_weights(layer);
    if (s != CS_OK) return s;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    if (!aligned16(h) || !aligned16(out) || (residual != nullptr && !aligned16(residual))) return CS_ERR_UNSUPPORTED;
    return exec_dispatch(plan, layer, h, support, B, residual, out, true, static_cast<cudaStream_t>(stream));
}

cs_status cs_bucket(cs_plan *plan, const int32_t *support, int32_t B, int32_t *counts, int32_t *offsets,
                    int32_t *token_ids, void *stream) {
    if (plan == nullptr || support == nullptr || counts == nullptr || offsets == nullptr || token_ids == nullptr)
        return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cs_status s = launch_check_support(plan, support, B, st);
    if (s != CS_OK) return s;
    return launch_bucket(plan, support, B, st, counts, offsets, token_ids);
}

// One step on the tensor cores: the sketch launch also splits the activations, the recovery runs inside the gate/up
// launch (or, for k beyond its list form, as a launch in front of it).
static cs_status decode_step(cs_plan *plan, const cs_layer *layer, const float *x, int B, RecoverOptions &o, float *x_out,
                             int32_t *sup, float *z, float *resid, cudaStream_t st) {
    const float *residual = layer->add_residual ? x : nullptr;
    o.decode = true; o.norm = layer->rms_gamma != nullptr;
    cs_status s = launch_sketch_slices(plan, layer, x, B, st);
    if (s != CS_OK) return s;
    if (decode_recovers(plan)) {
        const RecoverArgs ra = recover_args(plan, layer->Phi, layer->mu, plan->y_buf, B, sup, z, resid, o);
        return launch_decode_ffn(plan, layer, B, &ra, false, o.norm, residual, x_out, st);
    }
    s = launch_recover(plan, layer->Phi, layer->mu, plan->y_buf, B, sup, z, resid, true, st, o);
    if (s != CS_OK) return s;
    return launch_decode_ffn(plan, layer, B, nullptr, false, o.norm, residual, x_out, st);
}

cs_status cs_layer_step(cs_plan *plan, const cs_layer *layer, const float *x, int32_t B, float *x_out,
                        int32_t *support_out, float *z_out, float *resid_out, void *stream) {
    if (plan == nullptr || x == nullptr || x_out == nullptr) return CS_ERR_NULL;
    cs_status s = check_weights(layer);
    if (s != CS_OK) return s;
    if (layer->S == nullptr || layer->Phi == nullptr) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    if (!isfinite(layer->mu) || !(layer->mu > 0.f)) return CS_ERR_NONFINITE;
    if (!aligned16(x) || !aligned16(x_out) || !aligned16(layer->S) ||
        (layer->rms_gamma != nullptr && !aligned16(layer->rms_gamma)))
        return CS_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool norm = layer->rms_gamma != nullptr;
    const float *n = norm ? plan->n_buf : x;
    int32_t *sup = support_out != nullptr ? support_out : plan->sup_buf;
    if (use_decode_mma(plan, B)) {
        RecoverOptions o;
        return decode_step(plan, layer, x, B, o, x_out, sup, z_out, resid_out, st);
    }
    const bool gather = !plan->mma_ok || B < plan->mma_min_tokens;
    if (gather && plan->speculative && sketch_recover_ok(plan) && !plan->timing) {
        // Opt-in (cs_plan_set_speculative): sketch and recovery in one launch, and the gather FFN behind it
        // starts its weight stream on the first iterate while the other iterations run.  (Not while stages
        // are being timed: event records between the launches would serialise them.)
        if (plan->speculative == 2) {
            // L2 warm-up only: the plain gather kernel, which asks L2 for the first iterate's blocks before it
            // waits for the final supports
            s = launch_sketch_recover(plan, layer, x, B, plan->y_buf, norm ? plan->n_buf : nullptr, sup, z_out, resid_out, st);
            if (s != CS_OK) return s;
            return launch_ffn_gather(plan, layer, n, sup, B, layer->add_residual ? x : nullptr, x_out, false, st, plan->slot_table);
        }
        s = launch_sketch_recover(plan, layer, x, B, plan->y_buf, norm ? plan->n_buf : nullptr, support_out, z_out, resid_out, st);
        if (s != CS_OK) return s;
        return launch_ffn_gather_spec(plan, layer, n, B, layer->add_residual ? x : nullptr, x_out, st);
    }
    if (B <= plan->sense_tokens) {
        s = launch_sense_recover(plan, layer->S, layer->Phi, layer->mu, x, layer->rms_gamma, B, norm ? plan->n_buf : nullptr, sup, z_out,
                                 resid_out, st);
    } else {
        s = launch_sketch(plan, layer->S, x, layer->rms_gamma, B, plan->y_buf, norm ? plan->n_buf : nullptr, layer->Phi, layer->mu, st);
        if (s == CS_OK) s = launch_recover(plan, layer->Phi, layer->mu, plan->y_buf, B, sup, z_out, resid_out, true, st);
    }
    if (s != CS_OK) return s;
    // supports produced by the recovery are valid by construction: no device check here
    return exec_dispatch(plan, layer, n, sup, B, layer->add_residual ? x : nullptr, x_out, false, st);
}

cs_status cs_layer_step_ex(cs_plan *plan, const cs_layer *layer, const float *x, int32_t B,
                           const cs_step_options *opt, float *x_out, int32_t *support_out, float *z_out,
                           float *resid_out, void *stream) {
    if (opt == nullptr) return cs_layer_step(plan, layer, x, B, x_out, support_out, z_out, resid_out, stream);
    if (plan == nullptr || x == nullptr || x_out == nullptr) return CS_ERR_NULL;
    cs_status s = check_weights(layer);
    if (s != CS_OK) return s;
    const bool srht = opt->srht_sign != nullptr;
    if (layer->Phi == nullptr || (!srht && layer->S == nullptr)) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    if (!isfinite(layer->mu) || !(layer->mu > 0.f)) return CS_ERR_NONFINITE;
    if (!aligned16(x) || !aligned16(x_out) || (!srht && !aligned16(layer->S)) ||
        (layer->rms_gamma != nullptr && !aligned16(layer->rms_gamma)))
        return CS_ERR_UNSUPPORTED;
    s = check_options(plan, opt, true);
    if (s != CS_OK) return s;
    const bool norm = layer->rms_gamma != nullptr;
    if (srht && norm) return CS_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const float *n = norm ? plan->n_buf : x;
    const float *residual = layer->add_residual ? x : nullptr;
    if (opt->reuse_support) {   // no estimation this step: the previous supports execute
        s = launch_check_support(plan, opt->support_prev, B, st);
        if (s != CS_OK) return s;
        if (norm) {   // the sketch kernel also forms the normalised input
            s = launch_sketch(plan, layer->S, x, layer->rms_gamma, B, plan->y_buf, plan->n_buf, nullptr, 0.f, st);
            if (s != CS_OK) return s;
        }
        if (support_out != nullptr)
            CS_CUDA_TRY(plan, cudaMemcpyAsync(support_out, opt->support_prev, (size_t)B * plan->cfg.k * sizeof(int32_t),
                                              cudaMemcpyDeviceToDevice, st));
        return exec_dispatch(plan, layer, n, opt->support_prev, B, residual, x_out, false, st);
    }
    int32_t *sup = support_out != nullptr ? support_out : plan->sup_buf;
    if (use_decode_mma(plan, B) && !srht && opt->solver == CS_SOLVER_IHT) {   // as in cs_layer_step
        RecoverOptions o = iht_options(plan, opt);
        return decode_step(plan, layer, x, B, o, x_out, sup, z_out, resid_out, st);
    }
    if (B <= plan->sense_tokens && !srht && opt->solver == CS_SOLVER_IHT) {
        s = launch_sense_recover(plan, layer->S, layer->Phi, layer->mu, x, layer->rms_gamma, B, norm ? plan->n_buf : nullptr, sup, z_out,
                                 resid_out, st, iht_options(plan, opt));
        if (s != CS_OK) return s;
        return exec_dispatch(plan, layer, n, sup, B, residual, x_out, false, st);
    }
    if (srht) s = launch_sketch_srht(plan, opt->srht_sign, opt->srht_rows, x, B, plan->y_buf, st);
    else s = launch_sketch(plan, layer->S, x, layer->rms_gamma, B, plan->y_buf, norm ? plan->n_buf : nullptr, layer->Phi,
                           layer->mu, st);
    if (s != CS_OK) return s;
    s = recover_with(plan, layer->Phi, layer->mu, plan->y_buf, B, opt, sup, z_out, resid_out, !srht, st);
    if (s != CS_OK) return s;
    return exec_dispatch(plan, layer, n, sup, B, residual, x_out, false, st);
}

cs_status cs_layer_step_fallback(cs_plan *plan, cs_plan *dense, const cs_layer *layer, const float *x, int32_t B,
                                 const cs_step_options *opt, float tau, float *x_out, int32_t *support_out,
                                 float *z_out, float *resid_out, int32_t *flags_out, int32_t *n_fallback,
                                 void *stream) {
    if (plan == nullptr || dense == nullptr || n_fallback == nullptr) return CS_ERR_NULL;
    const cs_config &a = plan->cfg, &b = dense->cfg;
    if (a.d != b.d || a.d_ff != b.d_ff || a.group != b.group || a.m != b.m || a.w_dtype != b.w_dtype || b.k < a.k ||
        B > b.max_tokens)
        return CS_ERR_SHAPE;
    if (!isfinite(tau) || tau < 0.f) return CS_ERR_NONFINITE;
    if (opt != nullptr && opt->reuse_support) return CS_ERR_UNSUPPORTED;
    if (x_out == x) return CS_ERR_UNSUPPORTED;   // the second pass reads x again
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    float *resid = resid_out != nullptr ? resid_out : plan->resid_buf;
    cs_status s = cs_layer_step_ex(plan, layer, x, B, opt, x_out, support_out, z_out, resid, stream);
    if (s != CS_OK) return s;
    s = launch_confidence(plan, plan->y_buf, resid, B, tau, flags_out != nullptr ? flags_out : plan->fb_flags, plan->fb_list,
                          plan->fb_count, st);
    if (s != CS_OK) return s;
    int32_t n_low = 0;
    CS_CUDA_TRY(plan, cudaMemcpyAsync(&n_low, plan->fb_count, sizeof n_low, cudaMemcpyDeviceToHost, st));
    CS_CUDA_TRY(plan, cudaStreamSynchronize(st));
    *n_fallback = n_low;
    if (n_low == 0) return CS_OK;
    // the untrusted tokens alone, through the denser plan, and back into their rows
    s = launch_gather_rows(plan, x, plan->fb_list, n_low, dense->x_host_in, st);
    if (s != CS_OK) return s;
    cs_step_options second;
    memset(&second, 0, sizeof second);
    second.T = -1;
    if (opt != nullptr) { second.solver = opt->solver; second.srht_sign = opt->srht_sign; second.srht_rows = opt->srht_rows; }
    if (second.solver == CS_SOLVER_OMP && b.k > 64) second.solver = CS_SOLVER_IHT;
    s = cs_layer_step_ex(dense, layer, dense->x_host_in, n_low, &second, dense->x_host_out, nullptr, nullptr, nullptr, stream);
    if (s != CS_OK) return s;
    return launch_scatter_rows(plan, dense->x_host_out, plan->fb_list, n_low, x_out, st);
}

cs_status cs_layer_step_host(cs_plan *plan, const cs_layer *layer, const float *x_host, int32_t B,
                             float *x_out_host, int32_t *support_host, void *stream) {
    if (plan == nullptr || x_host == nullptr || x_out_host == nullptr) return CS_ERR_NULL;
    if (B <= 0 || B > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t bytes = (size_t)B * plan->cfg.d * sizeof(float);
    // validate before the first copy so that nothing is enqueued on an error
    cs_status s = check_weights(layer);
    if (s != CS_OK) return s;
    if (layer->S == nullptr || layer->Phi == nullptr) return CS_ERR_NULL;
    if (!isfinite(layer->mu) || !(layer->mu > 0.f)) return CS_ERR_NONFINITE;
    // Small transfers from and to page-locked memory: the copy engine's set-up costs as much as the
    // transfer or more, so a kernel of the launch chain fetches x over the bus and the last kernel of
    // the step stores the result straight into the caller's buffer.  Anything else goes through the
    // copy engine.  (Tensor-core batches, beyond 256 tokens too: d = 2048, 300 tokens 224 us a call against 300 through the copy
    // engine, 1000 tokens of d = 1024 315 against 415.)
    const float *x_alias = nullptr;
    float *out_alias = nullptr;
    if (bytes <= (plan->mma_ok && B >= plan->mma_min_tokens ? kZeroCopyBytesLarge : kZeroCopyBytes)) {
        x_alias = static_cast<const float *>(device_alias(x_host));
        out_alias = static_cast<float *>(device_alias(x_out_host));
        if (x_alias == nullptr || out_alias == nullptr || !aligned16(x_alias) || !aligned16(out_alias)) x_alias = nullptr;
    }
    if (x_alias != nullptr) {
        const int n4 = (int)(bytes / 16);
        launch_pdl(true, stage_in_kernel, dim3((n4 + 255) / 256), dim3(256), 0, st,
                   reinterpret_cast<const float4 *>(x_alias), reinterpret_cast<float4 *>(plan->x_host_in), n4);
        plan->launches++;
        CS_CUDA_TRY(plan, cudaGetLastError());
        s = cs_layer_step(plan, layer, plan->x_host_in, B, out_alias, support_host != nullptr ? plan->sup_buf : nullptr, nullptr,
                          nullptr, stream);
        if (s != CS_OK) return s;
    } else {
        CS_CUDA_TRY(plan, cudaMemcpyAsync(plan->x_host_in, x_host, bytes, cudaMemcpyHostToDevice, st));
        s = cs_layer_step(plan, layer, plan->x_host_in, B, plan->x_host_out, support_host != nullptr ? plan->sup_buf : nullptr,
                          nullptr, nullptr, stream);
        if (s != CS_OK) return s;
        CS_CUDA_TRY(plan, cudaMemcpyAsync(x_out_host, plan->x_host_out, bytes, cudaMemcpyDeviceToHost, st));
    }
    if (support_host != nullptr)
        CS_CUDA_TRY(plan, cudaMemcpyAsync(support_host, plan->sup_buf, (size_t)B * plan->cfg.k * sizeof(int32_t),
                                          cudaMemcpyDeviceToHost, st));
    return CS_OK;
}

cs_status cs_plan_set_crossover(cs_plan *plan, int32_t tokens) {
    if (plan == nullptr) return CS_ERR_NULL;
    if (tokens < 1 || tokens > 129) return CS_ERR_SHAPE;
    plan->mma_min_tokens = tokens;
    return CS_OK;
}

int32_t cs_plan_crossover(const cs_plan *plan) { return plan != nullptr ? plan->mma_min_tokens : 0; }

cs_status cs_plan_set_speculative(cs_plan *plan, int32_t on) {
    if (plan == nullptr) return CS_ERR_NULL;
    if (on && !sketch_recover_ok(plan)) return CS_ERR_UNSUPPORTED;
    if (on < 0 || on > 2) return CS_ERR_SHAPE;
    plan->speculative = on;
    return CS_OK;
}

cs_status cs_plan_enable_timing(cs_plan *plan, int32_t on) {
    if (plan == nullptr) return CS_ERR_NULL;
    plan->timing = on != 0;
    for (int i = 0; i < CS_STAGE_COUNT; ++i) plan->stage_seen[i] = 0;
    return CS_OK;
}

cs_status cs_plan_stage_times(cs_plan *plan, void *stream, float ms[CS_STAGE_COUNT]) {
    if (plan == nullptr || ms == nullptr) return CS_ERR_NULL;
    CS_CUDA_TRY(plan, cudaStreamSynchronize(static_cast<cudaStream_t>(stream)));
    for (int i = 0; i < CS_STAGE_COUNT; ++i) {
        ms[i] = 0.f;
        if (plan->stage_seen[i]) CS_CUDA_TRY(plan, cudaEventElapsedTime(&ms[i], plan->ev[2 * i], plan->ev[2 * i + 1]));
    }
    return CS_OK;
}

cs_status cs_prompt_support(cs_plan *plan, const float *S, const float *Phi, float mu, const void *H,
                            int32_t n, int32_t *support, float *z, float *resid, void *stream) {
    if (plan == nullptr || S == nullptr || Phi == nullptr || H == nullptr || support == nullptr) return CS_ERR_NULL;
    if (n <= 0 || n > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    if (!isfinite(mu) || !(mu > 0.f)) return CS_ERR_NONFINITE;
    if (!aligned16(S) || !aligned16(H)) return CS_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int blocks = 0;
    cs_status s = launch_prompt_colsum(plan, H, n, &blocks, st);
    if (s != CS_OK) return s;
    return launch_sense_recover(plan, S, Phi, mu, plan->colsum, nullptr, 1, nullptr, support, z, resid, st, RecoverOptions(), blocks, n);
}

cs_status cs_ffn_exec_shared(cs_plan *plan, const cs_layer *layer, const void *H, int32_t n,
                             const int32_t *support, void *out, void *stream) {
    if (plan == nullptr || H == nullptr || support == nullptr || out == nullptr) return CS_ERR_NULL;
    cs_status s = check_weights(layer);
    if (s != CS_OK) return s;
    if (n <= 0 || n > plan->cfg.max_tokens) return CS_ERR_SHAPE;
    if (!plan->mma_ok || !aligned16(H) || !aligned16(out)) return CS_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return launch_ffn_mma(plan, layer, H, nullptr, n, support, nullptr, plan->cfg.k, nullptr, nullptr, nullptr, out, st);   // checks the support
}

cs_status cs_last_device_status(cs_plan *plan, void *stream, int32_t *code) {
    if (plan == nullptr || code == nullptr) return CS_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    DeviceStatus hs;
    CS_CUDA_TRY(plan, cudaMemcpyAsync(&hs, plan->status, sizeof hs, cudaMemcpyDeviceToHost, st));
    CS_CUDA_TRY(plan, cudaMemsetAsync(plan->status, 0, sizeof hs, st));
    CS_CUDA_TRY(plan, cudaStreamSynchronize(st));
    *code = hs.code;
    return CS_OK;
}

int64_t cs_launch_count(const cs_plan *plan) { return plan != nullptr ? plan->launches : 0; }

const char *cs_last_cuda_error(const cs_plan *plan) { return plan != nullptr ? plan->cuda_error : ""; }

const char *cs_status_string(cs_status s) {
    switch (s) {
        case CS_OK: return "ok";
        case CS_ERR_NULL: return "null pointer";
        case CS_ERR_SHAPE: return "inconsistent shape";
        case CS_ERR_UNSUPPORTED: return "unsupported shape, dtype or alignment";
        case CS_ERR_SUPPORT: return "invalid support (must be ascending, distinct, in range)";
        case CS_ERR_NONFINITE: return "non-finite or non-positive scalar parameter";
        case CS_ERR_CUDA: return "CUDA runtime error";
        case CS_ERR_TIMEOUT: return "bounded device wait gave up";
    }
    return "unknown status";
}

}  // extern "C"
