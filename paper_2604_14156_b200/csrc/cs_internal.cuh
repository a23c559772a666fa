// Internal declarations shared by the library's translation units (not part of the C boundary).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cs.h"

namespace cs {

constexpr int kMaxG = 128;        // groups per layer
constexpr int kMaxM = 64;         // sketch rows
constexpr int kMaxD = 8192;       // hidden size
constexpr int kGatherThreads = 512;
constexpr int kGatherMaxRows = 160;  // channel rows one gather CTA owns at most (what its tables hold beside 192 KB of rings)
constexpr int kStaticMaxRows = 32;   // the same bound of the entry without a plan (part of its stated limit)
constexpr int kGatherMaxTokens = 16; // tokens per gather launch (scratch for partial sums)
constexpr int kSlotTableSlots = 32;  // slots per token of the recovery's slot table (small-batch step) ...
constexpr int kSlotTablePitch = 40;  // ... and ints per token: the slots, then a word that says "final"
constexpr int kReduceGroups = 32;    // partial-sum groups of the deterministic cross-CTA reduction
constexpr int kDecodeMaxTokens = 256;   // largest decode batch of exec_decode.cu; larger ones take the 128-token tiles of exec_mma.cu
constexpr int kMmaMinTokens = 16;    // decode batches at least this large always run on the tensor cores; a plan
                                     // lowers the bound by its G / k (cs_plan_set_crossover overrides it)

// Device status word values mirror cs_status (0 = ok).
struct DeviceStatus {
    int code;
};

}  // namespace cs

struct cs_plan {
    cs_config cfg;
    int G;
    int device;
    int sm_count;
    // device scratch
    float *n_buf;      // [max_tokens, d]  normalised FFN input
    float *y_buf;      // [max_tokens, m]
    int32_t *sup_buf;  // [max_tokens, k]
    float *partial;    // [kGatherMaxTokens, nx_max, d] partial down-projections of the gather path
    float *gram;       // [G, pitch] I - mu Phi^T Phi of the layer being mask_count, pitch = 32 ceil(G/32)
    float *resid_buf;     // [max_tokens] residual norms when the caller wants none (confidence fallback)
    int32_t *fb_flags;    // [max_tokens] confidence fallback: 1 = the token's recovery is not trusted
    int32_t *fb_list;     // [max_tokens] those tokens, ascending
    int32_t *fb_count;    // [1] their number
    int32_t *slot_table;  // [max_tokens, kSlotTablePitch] small-batch step: slot -> group of the recovery in flight
    unsigned *ticket;     // [max_tokens] arrival counters of the sketch CTAs (zero between launches)
    float *colsum;     // [kMeanRowBlocks, d] column sums of a prompt's hidden states, per block of rows
    cs::DeviceStatus *status;  // device status word
    // tensor-core path (bf16 weights, 128-channel groups, d a multiple of 256)
    uint32_t *mask;      // [max_tokens, 4] membership bits: bit g of token t
    unsigned *mask_count; // [1] decode batches: CTAs that have written their masks
    int32_t *counts;     // [G] tokens per group
    int32_t *offsets;    // [G + 1]
    int32_t *token_ids;  // [max_tokens * k] tokens of each group, ascending
    int32_t *glist;      // [G] groups with a non-empty bucket, ascending
    int32_t *nu;         // [1] their number
    void *x_bf16;        // [2][max_tokens, d] bf16 activations: rounded value, then remainder
    void *act;           // [2][max_tokens, d_ff] bf16 SwiGLU activations over the group list (value, remainder)
    float *mma_partial;  // [slices, padded tokens, d] f32 partial down projections
    int sense_tokens;    // up to this many tokens sensor and estimator are one launch (launch_sense_recover)
    int speculative;     // small batches, on the recovery's first iterate: 1 = start the weight stream, 2 = warm L2 only
    int mma_ok;          // shape qualifies for the tensor-core path
    int mma_min_tokens;  // smallest decode batch that takes it
    int last_slices;
    int pair_key_ng, pair_key_mtiles, pair_count;   // prompt gate/up: paired-tile count of the last shape seen
    int mma_slices;      // most list slices the down GEMM is split into
    float *x_host_in;  // [max_tokens, d] staging for the host-buffer entry point
    float *x_host_out; // [max_tokens, d]
    cudaEvent_t ev[2 * CS_STAGE_COUNT];  // start/stop per stage
    int timing;
    int stage_seen[CS_STAGE_COUNT];
    int nx_max;
    int64_t launches;
    char cuda_error[256];
};

namespace cs {

cs_status record_cuda(cs_plan *plan, cudaError_t e, const char *what);

#define CS_CUDA_TRY(plan, expr)                                                     \
    do {                                                                            \
        cudaError_t e_ = (expr);                                                    \
        if (e_ != cudaSuccess) return ::cs::record_cuda((plan), e_, #expr);         \
    } while (0)

// Brackets one stage's launches with events when timing is enabled.  On a capturing stream the
// records become event-record nodes of the graph (external events), which can be timed after a
// replay and cost far less than a record issued from the host between two launches.
struct StageTimer {
    cs_plan *p; int stage; cudaStream_t st;
    static void record(cudaEvent_t ev, cudaStream_t s) {
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusActive)
            cudaEventRecordWithFlags(ev, s, cudaEventRecordExternal);
        else
            cudaEventRecord(ev, s);
    }
    StageTimer(cs_plan *plan, int s, cudaStream_t stream) : p(plan), stage(s), st(stream) {
        if (p->timing) record(p->ev[2 * stage], st);
    }
    ~StageTimer() {
        if (p->timing) { record(p->ev[2 * stage + 1], st); p->stage_seen[stage] = 1; }
    }
};

// Kernel launchers (each enqueues on `st`, bumps plan->launches, returns a status).
// Phi != NULL: the launch also forms the recovery's matrix I - mu Phi^T Phi (plan->gram) in spare CTAs.
cs_status launch_sketch(cs_plan *plan, const float *S, const float *x, const float *gamma, int B,
                        float *y, float *n_out, const float *Phi, float mu, cudaStream_t st);
// The sensor in front of launch_decode_ffn: partial sketches per slice of columns (and of the squares, for the RMSNorm),
// the two bf16 token matrices, and plan->gram.  The recovery adds the partials up.
cs_status launch_sketch_slices(cs_plan *plan, const cs_layer *L, const float *x, int B, cudaStream_t st);
// The sketch of a token as launch_sketch_slices leaves it: partial sums per slice of 64 columns.
struct SketchParts {
    const float *y, *ss;       // [slices][B, m] and, with an RMSNorm, of the squares [slices][B]
    int slices, B, d;
    float eps;
    float *y_out;              // [B, m]
};
struct RecoverArgs {
    const float *Phi, *gram, *y;
    float mu, tgamma;          // tgamma = 2 mu gamma of the temporal term
    int m, G, k, T, B;
    int32_t *support;
    float *z, *resid;
    const int32_t *sup0; const float *z0;
    const int32_t *sup_prev; const float *z_prev;
    const int32_t *check;
    int32_t *delta; float *drift;
    uint32_t *mask;
    unsigned *mask_count;      // decode batches: counts the CTAs whose recoveries are done
    SketchParts parts;
    cs::DeviceStatus *status;
};
struct RecoverOptions {
    int T = -1;                                             // iterations; < 0: the plan's
    const int32_t *sup0 = nullptr; const float *z0 = nullptr;   // warm start
    float gamma = 0.f;                                      // temporal term towards (sup_prev, z_prev)
    const int32_t *sup_prev = nullptr; const float *z_prev = nullptr;
    const int32_t *check = nullptr;                         // supports to validate (ascending, distinct, in range) ...
    int32_t *delta = nullptr; float *drift = nullptr;       // ... and the drift of the result against them
    // launch_sketch_slices came before and the decode GEMMs come next: take the sketch from the partials (writing it to
    // plan->y_buf; norm: with the RMSNorm's row scale) and write the membership masks (plan->mask).
    bool decode = false, norm = false;
};
RecoverArgs recover_args(const cs_plan *plan, const float *Phi, float mu, const float *y, int B, int32_t *support, float *z,
                         float *resid, const RecoverOptions &o);
// gram_ready: plan->gram already holds this Phi's matrix (the sketch launch before formed it).
cs_status launch_recover(cs_plan *plan, const float *Phi, float mu, const float *y, int B,
                         int32_t *support, float *z, float *resid, bool gram_ready, cudaStream_t st,
                         const RecoverOptions &opt = RecoverOptions());
// Sensor and estimator in one launch, a cluster of CTAs per token, for at most plan->sense_tokens tokens.  blocks > 0: one
// token whose x is the sum of `blocks` rows [blocks, d] divided by n (a prompt's mean hidden state).
constexpr int kSenseMaxTokens = 16;   // bound of plan->sense_tokens, see recover.cu
cs_status launch_sense_recover(cs_plan *plan, const float *S, const float *Phi, float mu, const float *x, const float *gamma, int B,
                               float *n_out, int32_t *support, float *z, float *resid, cudaStream_t st,
                               const RecoverOptions &opt = RecoverOptions(), int blocks = 0, int n = 1);
// the other estimators (solvers.cu)
cs_status prepare_solvers(cs_plan *plan);
cs_status launch_niht(cs_plan *plan, const float *Phi, float mu_fallback, const float *y, int B, int T,
                      int32_t *support, float *z, float *resid, cudaStream_t st);
cs_status launch_omp(cs_plan *plan, const float *Phi, const float *y, int B, int32_t *support, float *z, float *resid,
                     cudaStream_t st);
// the structured sketch (srht.cu)
cs_status launch_sketch_srht(cs_plan *plan, const uint32_t *sign_bits, const int32_t *rows, const float *h, int B, float *y,
                             cudaStream_t st);
// check: validate the supports on the device (ascending, distinct, in range) inside the same launch.
// warm: slot tables of a recovery still running in the launch ahead (launch_sketch_recover); the kernel
// asks L2 for the weight blocks they name before it waits for the final supports.
cs_status launch_ffn_gather(cs_plan *plan, const cs_layer *layer, const float *h, const int32_t *support,
                            int B, const float *residual, float *out, bool check, cudaStream_t st,
                            const int32_t *warm = nullptr);
// The small-batch step: sketch and recovery in one launch, whose programmatic trigger fires when the
// first iterate's slot table is in memory; the gather FFN launched behind it starts on that table,
// follows the table while the iteration runs, and settles on the final one.
bool sketch_recover_ok(const cs_plan *plan);
cs_status prepare_sketch(cs_plan *plan);
cs_status launch_sketch_recover(cs_plan *plan, const cs_layer *L, const float *x, int B, float *y, float *n_out,
                                int32_t *support, float *z, float *resid, cudaStream_t st);
cs_status launch_ffn_gather_spec(cs_plan *plan, const cs_layer *layer, const float *h, int B, const float *residual,
                                 float *out, cudaStream_t st);
cs_status prepare_ffn_gather(cs_plan *plan);
cs_status launch_support_drift(cs_plan *plan, const int32_t *prev, const int32_t *cur, int B, int32_t *drift,
                               float *ratio, cudaStream_t st);
// confidence fallback (control.cu): flags tokens whose relative residual exceeds tau, lists them, moves rows
cs_status launch_confidence(cs_plan *plan, const float *y, const float *resid, int B, float tau, int32_t *flags,
                            int32_t *list, int32_t *count, cudaStream_t st);
cs_status launch_gather_rows(cs_plan *plan, const float *src, const int32_t *list, int n, float *dst, cudaStream_t st);
cs_status launch_scatter_rows(cs_plan *plan, const float *src, const int32_t *list, int n, float *dst, cudaStream_t st);
cs_status launch_uds_budget(cs_plan *plan, const float *logits, int B, int V, float m_base, float gamma,
                            int m_min, int m_max, float *H, int32_t *m_t, cudaStream_t st);
cs_status launch_check_support(cs_plan *plan, const int32_t *support, int B, cudaStream_t st);
cs_status prepare_ffn_mma(cs_plan *plan);
cs_status launch_bucket(cs_plan *plan, const int32_t *support, int B, cudaStream_t st, int32_t *counts = nullptr,
                        int32_t *offsets = nullptr, int32_t *token_ids = nullptr);
cs_status launch_split_bf16(cs_plan *plan, const float *x, void *y_hi, void *y_lo, size_t n, cudaStream_t st);
cs_status launch_ffn_mma(cs_plan *plan, const cs_layer *L, const void *X, const void *X_lo, int M, const int32_t *glist,
                         const int32_t *ng_dev, int ng_host, const uint32_t *mask, const float *residual,
                         float *out_f32, void *out_bf16, cudaStream_t st);
// decode batches of at most kDecodeMaxTokens tokens on the tensor cores (exec_decode.cu)
cs_status prepare_decode(cs_plan *plan);
int decode_slices(const cs_plan *plan);
cs_status launch_decode_prep(cs_plan *plan, const float *h, const int32_t *support, int B, bool check, cudaStream_t st);
// recover != NULL and decode_recovers(): the recovery runs inside the gate/up launch; otherwise the launches before have
// left the masks (plan->mask); given: they are those of supports the caller gave (launch_decode_prep).  norm: the row scales come from the sketch's partial squares.
bool decode_recovers(const cs_plan *plan);
cs_status launch_decode_ffn(cs_plan *plan, const cs_layer *L, int B, const RecoverArgs *recover, bool given, bool norm,
                            const float *residual, float *out, cudaStream_t st);
// Column sums of H per block of rows (plan->colsum); *blocks = their number.
constexpr int kMeanRowBlocks = 16;
cs_status prepare_prompt(cs_plan *plan);
cs_status launch_prompt_colsum(cs_plan *plan, const void *H, int n, int *blocks, cudaStream_t st);

// Programmatic dependent launch: a kernel launched through launch_pdl may start while its
// predecessor in the stream is still running (its CTAs become resident, run their prologue and
// then block in pdl_wait until the predecessor's writes are complete and visible).  Kernels call
// pdl_launch_dependents early so that their successor can do the same.  Both are no-ops for a
// kernel launched the ordinary way (pdl = false).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Loads of data that the kernel before this one produced.  They are volatile asm statements, like
// the wait itself, so the compiler keeps them after it; a plain load through a const __restrict__
// pointer (or __ldg) may be turned into a non-coherent load and moved above the wait, which reads
// what the buffer held before (seen as rare wrong recoveries when a plan's scratch was reused).
__device__ __forceinline__ float ld_dep(const float *p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ int ld_dep(const int32_t *p) {
    int v;
    asm volatile("ld.global.s32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_dep4(const float *p) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// The partial sketches share plan->mma_partial with the down GEMM, whose first store comes after the recovery:
// y [d / 64][B, m], then the squares [d / 64][B].  (d / 64) (m + 1) B <= 2 d B floats.
inline float *sketch_partials(const cs_plan *plan) { return plan->mma_partial; }
inline float *sketch_square_partials(const cs_plan *plan, int B) {
    return plan->mma_partial + (size_t)(plan->cfg.d / 64) * B * plan->cfg.m;
}

// The small kernels around the large ones ask for the large ones' split of L1 and shared memory.  An SM changes its split
// only when it is empty, so with the default split a CTA of 200 KB does not start beside a running recovery: at 64
// tokens half of the gate/up CTAs then began 12 us late, when the last recovery on their SM had ended.
template <typename Fn> inline cudaError_t prefer_shared(Fn *kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
}
cs_status prepare_recover(cs_plan *plan);

// ---- small device helpers -------------------------------------------------------------------
// Rows 2*blk and 2*blk+1 of M = I - mu Phi^T Phi by a CTA of kGramThreads threads.  M is stored
// row-major with a pitch of 32 * ceil(G / 32) floats, the columns past G zero, so that a recovery
// thread can read its row with aligned 16-byte loads and needs no bounds in its inner loop.
// The values depend on parameters only and are computed at once; the store waits for the kernels
// before this one, which may still be reading the previous layer's matrix.
constexpr int kGramThreads = 256;
inline int gram_blocks(int G) { return (G + 1) / 2; }
__host__ __device__ inline int gram_pitch(int G) { return (G + 31) & ~31; }
__device__ __forceinline__ void gram_rows(const float *__restrict__ Phi, float mu, int m, int G, int blk,
                                          float *__restrict__ gram) {
    const int a = blk * 2 + (threadIdx.x >> 7), b = threadIdx.x & 127;
    const int pitch = gram_pitch(G);
    const bool valid = a < G && b < G;
    float s0 = 0.f, s1 = 0.f;
    if (valid) {
        int i = 0;
        for (; i + 1 < m; i += 2) {
            s0 = fmaf(__ldg(Phi + i * G + a), __ldg(Phi + i * G + b), s0);
            s1 = fmaf(__ldg(Phi + (i + 1) * G + a), __ldg(Phi + (i + 1) * G + b), s1);
        }
        if (i < m) s0 = fmaf(__ldg(Phi + i * G + a), __ldg(Phi + i * G + b), s0);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (a < G && b < pitch) gram[a * pitch + b] = valid ? (a == b ? 1.f : 0.f) - mu * (s0 + s1) : 0.f;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// L2 policy of the weights, which are read once: first to leave L2, so that they do not push out the activations, S and
// Phi, and the kernels' own code, which after a 270 MB step without this is fetched from HBM again (7B step at 64
// tokens 63.8 -> 60.0 us; 200 tokens 135 -> 121 in bursts of a few ms, no gain over a second of load).
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// Four floats as bf16 values and bf16 remainders: hi = round(x), lo = round(x - hi).
__device__ __forceinline__ void split4(float a, float b, float c, float e, uint2 &hi, uint2 &lo) {
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(a, b), h1 = __floats2bfloat162_rn(c, e);
    const __nv_bfloat162 l0 = __floats2bfloat162_rn(a - __low2float(h0), b - __high2float(h0));
    const __nv_bfloat162 l1 = __floats2bfloat162_rn(c - __low2float(h1), e - __high2float(h1));
    hi.x = *reinterpret_cast<const uint32_t *>(&h0); hi.y = *reinterpret_cast<const uint32_t *>(&h1);
    lo.x = *reinterpret_cast<const uint32_t *>(&l0); lo.y = *reinterpret_cast<const uint32_t *>(&l1);
}

__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// Widen one 16-byte chunk of weights to floats: 8 values for bf16, 4 for f32.
template <typename WT> struct Chunk;
template <> struct Chunk<__nv_bfloat16> {
    static constexpr int kElems = 8;
    __device__ static __forceinline__ void widen(const uint4 &q, float (&f)[8]) {
        f[0] = bf16_lo(q.x); f[1] = bf16_hi(q.x); f[2] = bf16_lo(q.y); f[3] = bf16_hi(q.y);
        f[4] = bf16_lo(q.z); f[5] = bf16_hi(q.z); f[6] = bf16_lo(q.w); f[7] = bf16_hi(q.w);
    }
};
template <> struct Chunk<float> {
    static constexpr int kElems = 4;
    __device__ static __forceinline__ void widen(const uint4 &q, float (&f)[4]) {
        f[0] = __uint_as_float(q.x); f[1] = __uint_as_float(q.y);
        f[2] = __uint_as_float(q.z); f[3] = __uint_as_float(q.w);
    }
};

}  // namespace cs
