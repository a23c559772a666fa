// Actuator, tensor-core regime for decode batches of at most kDecodeMaxTokens tokens with independent supports.
//
//   decode_gateup_kernel, decode_gateup_pair_kernel
//                          act[t, c] = silu(n_t . W_gate[c]) (n_t . W_up[c]) for every token t and channel c, in its support
//                          or not
//   decode_down_kernel     partial[z, t, :] = sum over the channels of list slice z that are in t's support of
//                          act[t, c] Wd_t[c, :]
//   decode_reduce_kernel   out = residual + sum_z partial
//
// Both GEMMs put the tokens on the M side of the MMA and stream the weights as its N operand: at these batch sizes
// the step is bound by the weight bytes (HBM), and what limits a kernel before that is shared memory, which every
// byte crosses once when TMA writes it and once per instruction that reads it.  As the N operand a weight
// byte is read by one instruction per 128 token rows; with the weights on the M side (128 rows per instruction,
// gate and up apart, the token operand read by both) a k block of 32 KB of weights cost 112 KB of shared-memory
// traffic, here 20 KB of weights cost 72 KB.
//
// f32 activations enter as two bf16 matrices, rounded value and remainder (16 mantissa bits together).  PACK
// (at most 64 tokens): values are rows 0.. and remainders rows 64.. of ONE 128-row operand, their products are added in
// the epilogue.  Otherwise values and remainders are two operands that accumulate into the same tensor-memory
// columns; MT = 2 (more than 128 tokens) keeps two accumulators (gate/up of a step with at most 64 groups per token runs on pairs of
// CTAs there).  Rows no token owns hold whatever shared memory held: rows of an MMA do not mix, and those results are never read.
//
// Balance: the channel tiles of gate/up are not tied to the 128-channel groups.  A CTA takes R channels, R the
// multiple of 8 that gives every SM one CTA (80 at d_ff = 11008: 138 CTAs on 148 SMs; one CTA per group left 62 SMs
// without work and took 39.7 us for 180 MB at 64 tokens).  The down GEMM has d / 256 column tiles times
// as many list slices as fill the SMs, cut at 64-channel k blocks.
//
// Supports: in a step gate/up computes every channel of every token and the down GEMM leaves out what a token's support does not
// hold, by the instruction's lane mask (lanes = tokens, so a k block's mask is its group's membership bits; the
// accumulators are zeroed first and only ever added to).  So nothing waits for the recovery before the down GEMM,
// and the recovery runs inside the gate/up launch, in four warps of each CTA that take the tokens in turn.
// A step is then sketch -> gate/up (+ recovery) -> down -> reduction, each started early (programmatic dependent
// launch) and streaming its weights before it waits for what the launch before produces.  With the recovery as a launch
// ahead of gate/up the weight stream began 5.4 us after the step, in this form while the sketch still runs.
// What an earlier launch of the step wrote is read behind a launch's own wait, since a trigger orders nothing in memory.  The
// one exception are the masks in the down launch: the CTAs that write them count themselves (release), and a down CTA that finds
// the count complete (acquire) may read them at once; one that does not waits first.  The reduction sets the count back.
#include "mma_core.cuh"
#include "recover_core.cuh"

namespace cs {

namespace {

constexpr int kEpiWarps = 8;                         // two per quarter of the tensor-memory lanes
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kDecThreads = 64 + kEpiThreads;        // + TMA warp, MMA warp
constexpr int kRecNW = kMaxG / 32, kRecThreads = 32 * kRecNW;   // the recovery's warps of a gate/up CTA
constexpr int kDecRing = 208 * 1024;                 // operand ring at most
constexpr int kDecMaxSlices = 20;
constexpr int kDecBN = 256;                          // output columns of a down tile

// How the token operand is laid out in a stage: boxes of `box` rows, `nbox` of them per matrix (value, remainder).
struct TokenTile {
    int box, nbox;
    int lo_off;       // byte offset of the remainder rows
    int bytes;        // of the whole operand in a stage
    int over;         // bytes past it that the last tile's MMA reads (rows no token owns)
};
__host__ __device__ inline TokenTile token_tile(bool pack, int mt, int B) {
    TokenTile t;
    t.over = 0;
    if (pack || mt == 1) {
        t.box = (B + 7) & ~7; t.nbox = 1;
        t.lo_off = pack ? kABytes / 2 : kABytes;
        t.bytes = pack ? kABytes : 2 * kABytes;
    } else {
        t.box = 64; t.nbox = (B + 63) / 64;
        t.lo_off = t.nbox * 64 * BK * 2;
        t.bytes = 2 * t.lo_off;
        t.over = (4 - t.nbox) * 64 * BK * 2;
    }
    return t;
}
__device__ __forceinline__ void load_tokens(const TokenTile &t, uint8_t *dst, const CUtensorMap *hi, const CUtensorMap *lo,
                                            int x, uint64_t *bar) {
    for (int i = 0; i < t.nbox; ++i) {
        tma_load_2d(dst + i * (64 * BK * 2), hi, x, i * 64, bar);
        tma_load_2d(dst + t.lo_off + i * (64 * BK * 2), lo, x, i * 64, bar);
    }
}
// Ring stages: [tokens][weights] each; what the MMA reads past the tokens of the last stage stays inside the ring.
__host__ __device__ inline int ring_stages(const TokenTile &t, int wbytes) {
    const int over = t.over > wbytes ? t.over - wbytes : 0, n = (kDecRing - over) / (t.bytes + wbytes);
    return n < kMaxStages ? n : kMaxStages;
}
__host__ __device__ inline int ring_bytes(const TokenTile &t, int wbytes) {
    return ring_stages(t, wbytes) * (t.bytes + wbytes) + (t.over > wbytes ? t.over - wbytes : 0);
}
// No more shared memory than the ring needs: the sketch of the step behind fits beside it.
inline size_t decode_smem(const TokenTile &t, int wbytes) { return 1024 + (size_t)ring_bytes(t, wbytes) + sizeof(Barriers); }
__device__ __forceinline__ int token_tx_bytes(const TokenTile &t) { return 2 * t.nbox * t.box * BK * 2; }

__device__ __forceinline__ void prefetch_map(const CUtensorMap *m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(m) : "memory");
}
// from L2: the kernel that wrote it may have run beside this one's predecessor on this SM
__device__ __forceinline__ uint4 ld_l2(const int32_t *p) {
    uint4 v;
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }

// This CTA's masks are written (and a barrier has joined the threads that wrote them).
__device__ __forceinline__ void count_masks(unsigned *mask_count) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(mask_count) : "memory");
}
// Union of the tokens' supports (their masks are visible): union_s, zero before the barrier that precedes the call, is
// complete behind the one that follows it.
__device__ __forceinline__ void collect_union(const int32_t *mask, int B, uint32_t *union_s) {
    for (int t = threadIdx.x; t < B; t += blockDim.x) {
        const uint4 m = ld_l2(mask + (size_t)t * 4);
        if (m.x) atomicOr(&union_s[0], m.x);
        if (m.y) atomicOr(&union_s[1], m.y);
        if (m.z) atomicOr(&union_s[2], m.z);
        if (m.w) atomicOr(&union_s[3], m.w);
    }
}
__device__ __forceinline__ int union_size(const uint32_t *u) { return __popc(u[0]) + __popc(u[1]) + __popc(u[2]) + __popc(u[3]); }
__device__ __forceinline__ int union_rank(const uint32_t *u, int g) {   // groups of the union below g
    int n = __popc(u[g >> 5] & ((1u << (g & 31)) - 1u));
    for (int w = 0; w < (g >> 5); ++w) n += __popc(u[w]);
    return n;
}

// The accumulator of one 128-row tile (columns tcol .. tcol + 16 nchunk) into shared memory, row-major with pitch P
// floats; `rows` rows are wanted (PACK: from each half).
template <bool PACK>
__device__ __forceinline__ void dump_tile(uint32_t tmem, int nchunk, float *dst, int P, int rows, int warp, int lane) {
    const int q = warp & 3, sub = (warp - 2) >> 2;
    const int row = q * 32 + lane;
    if ((PACK ? (q & 1) : q) * 32 >= rows) return;   // nobody's rows
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16);
    for (int c = sub; c < nchunk; c += kEpiWarps / 4) {
        uint32_t v[16];
        tc_ld16(tbase + c * 16, v);
        tc_wait_ld();
        float4 *o = reinterpret_cast<float4 *>(dst + (size_t)row * P + c * 16);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            o[j] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]), __uint_as_float(v[4 * j + 2]),
                               __uint_as_float(v[4 * j + 3]));
    }
}
template <bool PACK> __device__ __forceinline__ float4 row4(const float *s, int P, int r, int c) {
    float4 v = *reinterpret_cast<const float4 *>(s + (size_t)r * P + c);
    if (PACK) {
        const float4 w = *reinterpret_cast<const float4 *>(s + (size_t)(r + 64) * P + c);
        v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
    }
    return v;
}

// One k block of MMAs: token operand at a0 (remainders at a0 + lo_off) against the N operand given by bdesc(k4).
// lanes != NULL: the 128-bit lane mask of each 128-token tile (a set bit leaves that lane of the accumulator alone).
template <bool PACK, int MT, typename BDesc>
__device__ __forceinline__ void mma_kblock(uint32_t tmem, uint32_t a0, uint32_t lo_off, uint32_t idesc, bool first, BDesc bdesc,
                                           const uint4 *lanes = nullptr) {
#pragma unroll
    for (int k4 = 0; k4 < BK / 16; ++k4) {
        const uint64_t bd = bdesc(k4);
#pragma unroll
        for (int t = 0; t < MT; ++t) {
            const uint32_t a = a0 + t * kABytes + k4 * 32;
            if (lanes != nullptr) {
                tc_mma_lanes(tmem + t * 256, desc_sw128(a, 16), bd, idesc, lanes[t]);
                if (!PACK) tc_mma_lanes(tmem + t * 256, desc_sw128(a + lo_off, 16), bd, idesc, lanes[t]);
            } else {
                tc_mma(tmem + t * 256, desc_sw128(a, 16), bd, idesc, !first || k4 != 0);
                if (!PACK) tc_mma(tmem + t * 256, desc_sw128(a + lo_off, 16), bd, idesc, 1);
            }
        }
    }
}

// ---- gate / up ------------------------------------------------------------------------------------------
// CTA x: channels [x R, x R + R), and with KC > 0 (slots of the recovery's list form, in units of 8) the recovery of tokens
// x, x + gridDim.x, ...
// mask != NULL (KC == 0, MT == 2): the supports were given, and where it makes a CTA's share smaller the channels are those of
// the groups in use only, in units of 16 that the CTAs share evenly (tm_gu, tm_uu: the weights in boxes of 16 rows).  Groups outside
// the union keep what `act` held, and the down launch does not read them.
constexpr int kListRows = 16;
template <bool PACK, int MT, int KC>
__global__ void __launch_bounds__(kDecThreads + kRecThreads, 1)
decode_gateup_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_x_lo,
                     const __grid_constant__ CUtensorMap tm_g, const __grid_constant__ CUtensorMap tm_u,
                     const __grid_constant__ CUtensorMap tm_gu, const __grid_constant__ CUtensorMap tm_uu, int B, int R, int d, int d_ff,
                     const int32_t *mask, const float *ss_part, float eps, const __grid_constant__ RecoverArgs ra,
                     __nv_bfloat16 *__restrict__ act, __nv_bfloat16 *__restrict__ act_lo, DeviceStatus *status) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ float rscale_s[MT * BM];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const TokenTile tt = token_tile(PACK, MT, B);
    const int c0 = blockIdx.x * R;
    constexpr bool LIST = KC == 0 && MT == 2;
    __shared__ uint32_t union_s[LIST ? 4 : 1];
    __shared__ int unit_s[LIST ? BM / kListRows : 1];   // first channel of each unit of this CTA
    bool by_list = LIST && mask != nullptr;
    Barriers *bars = reinterpret_cast<Barriers *>(base + (by_list ? kDecRing : ring_bytes(tt, 2 * R * BK * 2)));
    const uint32_t tcols = MT == 2 ? 512u : 256u;
    const int kblocks = d / BK;
    if (threadIdx.x == 0) { prefetch_map(&tm_g); prefetch_map(&tm_u); prefetch_map(&tm_x); prefetch_map(&tm_x_lo); }
    if (by_list && threadIdx.x < 4) union_s[threadIdx.x] = 0u;
    setup_cta(bars, warp, tcols);
    int units = 0;
    if constexpr (LIST) {
        if (by_list) {
            pdl_wait();
            collect_union(mask, B, union_s);
            __syncthreads();
            constexpr int kUnits = 128 / kListRows;   // of a group
            const int total = union_size(union_s) * kUnits, per = (total + (int)gridDim.x - 1) / (int)gridDim.x;
            by_list = per * kListRows < R;
            if (by_list) {
                const int u0 = blockIdx.x * per, g = threadIdx.x;
                units = max(0, min(per, total - u0));
                if (g < kMaxG && ((union_s[g >> 5] >> (g & 31)) & 1u)) {
                    const int first = union_rank(union_s, g) * kUnits;
                    for (int u = max(first, u0); u < min(first + kUnits, u0 + units); ++u) unit_s[u - u0] = g * 128 + (u - first) * kListRows;
                }
                __syncthreads();
                R = units * kListRows;
                if (units == 0) { teardown_cta(bars, warp, tcols); return; }
            }
        }
    }
    const int wbytes = 2 * R * BK * 2;                   // gate rows then up rows
    const int stage_bytes = tt.bytes + wbytes;
    const int stages = ring_stages(tt, wbytes);

    if (warp == 0 && by_list) {   // lane u: the gate rows of unit u, lane 16 + u: its up rows (one lane for all: 47 ns a box)
        const int tx = wbytes + token_tx_bytes(tt), u = lane & 15;
        const uint64_t once = policy_evict_first();
        const CUtensorMap *tm_w = lane < 16 ? &tm_gu : &tm_uu;
        const int w_off = tt.bytes + (lane < 16 ? 0 : wbytes / 2) + u * (kListRows * BK * 2), ch = u < units ? unit_s[u] : 0;
        int s = 0, ph = 1;
        for (int kb = 0; kb < kblocks; ++kb) {
            bool ok = true;
            if (kb >= stages && lane == 0) ok = mbar_wait(&bars->empty[s], ph, bars, status);
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
            uint8_t *st = base + (size_t)s * stage_bytes;
            if (lane == 0) mbar_expect_tx(&bars->full[s], tx);
            __syncwarp();
            if (u < units) tma_load_2d(st + w_off, tm_w, kb * BK, ch, &bars->full[s], once);
            if (lane == 0) load_tokens(tt, st, &tm_x, &tm_x_lo, kb * BK, &bars->full[s]);
            if (++s == stages) { s = 0; ph ^= 1; }
        }
    } else if (warp == 0) {
        if (lane == 0) {
            const int tx = wbytes + token_tx_bytes(tt);
            const uint64_t once = policy_evict_first();
            auto load_w = [&](int kb, int s) {
                uint8_t *w = base + (size_t)s * stage_bytes + tt.bytes;
                tma_load_2d(w, &tm_g, kb * BK, c0, &bars->full[s], once);
                tma_load_2d(w + wbytes / 2, &tm_u, kb * BK, c0, &bars->full[s], once);
            };
            // weights are parameters: the first ring is requested before anything is waited for
            const int pre = min(stages, kblocks);
            for (int kb = 0; kb < pre; ++kb) { mbar_expect_tx(&bars->full[kb], tx); load_w(kb, kb); }
            pdl_wait();   // the token matrices
            for (int kb = 0; kb < pre; ++kb) load_tokens(tt, base + (size_t)kb * stage_bytes, &tm_x, &tm_x_lo, kb * BK, &bars->full[kb]);
            int s = 0, ph = 0;
            for (int kb = pre; kb < kblocks; ++kb) {
                if (!mbar_wait(&bars->empty[s], ph, bars, status)) break;
                mbar_expect_tx(&bars->full[s], tx);
                load_w(kb, s);
                load_tokens(tt, base + (size_t)s * stage_bytes, &tm_x, &tm_x_lo, kb * BK, &bars->full[s]);
                if (++s == stages) { s = 0; ph ^= 1; }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = make_idesc_rt(2 * R, false, false);
            const uint32_t tmem = bars->tmem_base;
            bool ok = true;
            int s = 0, ph = 0;
            for (int kb = 0; kb < kblocks; ++kb) {
                ok = mbar_wait(&bars->full[s], ph, bars, status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a0 = smem_u32(base + (size_t)s * stage_bytes), w0 = a0 + tt.bytes;
                mma_kblock<PACK, MT>(tmem, a0, tt.lo_off, idesc, kb == 0, [&](int k4) { return desc_sw128(w0 + k4 * 32, 16); });
                tc_commit(&bars->empty[s]);
                if (++s == stages) { s = 0; ph ^= 1; }
            }
            if (ok) tc_commit(&bars->acc_ready);
        }
    } else if (warp < kDecThreads / 32) {
        const int et = threadIdx.x - 64, r4 = R / 4;
        pdl_wait();   // the row squares; and nothing is stored before the kernels before this one are complete
        if (KC == 0) pdl_launch_dependents();
        for (int t = et; t < MT * BM; t += kEpiThreads) {
            float rs = 1.f;
            if (ss_part != nullptr && t < B) {
                float q = 0.f;
                for (int i = 0; i < d / 64; i += 16) {   // d is a multiple of 256
                    float v[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) v[u] = i + u < d / 64 ? ld_dep(ss_part + (size_t)(i + u) * B + t) : 0.f;
#pragma unroll
                    for (int u = 0; u < 16; ++u) q += v[u];
                }
                rs = rsqrtf(q / (float)d + eps);
            }
            rscale_s[t] = rs;
        }
        // one warp polls, the others sleep at the barrier behind it
        if (warp == 2) mbar_wait(&bars->acc_ready, 0, bars, status);
        epi_sync();
        const bool ok = *reinterpret_cast<volatile uint32_t *>(&bars->aborted) == 0u && mbar_wait(&bars->acc_ready, 0, bars, status);
        tc_fence_after();
        float *dump = reinterpret_cast<float *>(base);   // the ring is free: every load has been consumed
        const int P = ((2 * R + 31) & ~31) + 4;
#pragma unroll 1
        for (int t = 0; t < MT; ++t) {
            const int t0 = t * BM, rows = min(B - t0, PACK ? 64 : BM);
            if (t > 0) epi_sync();
            if (ok) dump_tile<PACK>(bars->tmem_base + t * 256, 2 * R / 16, dump, P, rows, warp, lane);
            epi_sync();
            if (ok) {
#pragma unroll 2
                for (int i = et; i < rows * r4; i += kEpiThreads) {
                    const int r = i / r4, c = (i - r * r4) * 4, ch = by_list ? unit_s[c / kListRows] + c % kListRows : c0 + c;
                    if (ch >= d_ff) continue;
                    const float4 g = row4<PACK>(dump, P, r, c), u = row4<PACK>(dump, P, r, R + c);
                    const float sc = rscale_s[t0 + r];
                    uint2 hi, lo;
                    split4(silu_f(g.x * sc) * (u.x * sc), silu_f(g.y * sc) * (u.y * sc), silu_f(g.z * sc) * (u.z * sc),
                           silu_f(g.w * sc) * (u.w * sc), hi, lo);
                    const size_t off = (size_t)(t0 + r) * d_ff + ch;
                    *reinterpret_cast<uint2 *>(act + off) = hi;
                    *reinterpret_cast<uint2 *>(act_lo + off) = lo;
                }
            }
        }
    } else if constexpr (KC > 0) {
        constexpr int kRecBar = 3;
        __shared__ RecoverSmem<kRecNW, KC> rs;
        const int g = threadIdx.x - kDecThreads;
        float phc[32];
        if (ra.m <= 32) recover_load_phi<kRecNW>(ra.Phi, ra.m, ra.G, g, phc);
        const GramSource M{ra.gram, gram_pitch(ra.G)};
        pdl_wait();   // the partial sketches and M come from the kernel before
        for (int t = blockIdx.x; t < B; t += gridDim.x) {
            recover_row<kRecNW, KC, kRecBar>(
                rs, ra, M, [&](auto &sm) { y_from_parts<kRecNW, kRecBar>(sm, ra.parts, g, t, ra.m); }, ra.mask, g, t, phc);
            bar_sync<kRecBar, kRecThreads>();
        }
        // this CTA's masks are written (the barrier that ends the loop, or no token at all)
        if (g == 0) {
            count_masks(ra.mask_count);
            pdl_launch_dependents();
        }
    }
    teardown_cta(bars, warp, tcols);
}

// The same for a step of more than 128 tokens and at most 64 groups per token, on pairs of CTAs (a cluster of two).  (Beyond 64 groups the
// recovery is a launch ahead and gate/up the kernel above with two accumulators, as with given supports.)  With both accumulators in one CTA every weight tile
// is read from shared memory by four instructions and every k block moves 228 KB through that port for 20 KB of weights (1.03 us a k
// block, 68 us at 7B and 200 tokens, the tensor pipe 51 % busy).  Here one instruction has M = 256: each CTA holds half of the tokens
// (their values and their remainders, 128 rows each) and half of the pair's channels, R of 2 R, gate rows then up rows: 156 KB for the
// same 20 KB of weights per CTA.  One step, 7B: 200 tokens 135.5 to 127.0 us, in short bursts 132 to 121, 256 tokens 139 to 127; d = 5120
// with 27 of 108 groups, 200 tokens 189 to 181; 129 tokens 113.9 to 112.6, so every such batch takes it.
// Gate accumulates in tensor-memory columns 0 .. 2 R, up from 256 on.  The even CTA's MMA thread issues for both; no multicast load, each
// CTA fetches its own tiles and signals the even CTA's barrier.
constexpr int kPairTokenBytes = 2 * kABytes;   // value rows, then remainder rows
__host__ __device__ inline int gateup_pair_stages(int R) { return min(kMaxStages, kDecRing / (kPairTokenBytes + 2 * R * BK * 2)); }
template <int KC>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kDecThreads + kRecThreads, 1)
decode_gateup_pair_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_x_lo,
                          const __grid_constant__ CUtensorMap tm_g, const __grid_constant__ CUtensorMap tm_u, int B, int half, int R, int d,
                          int d_ff, const float *ss_part, float eps, const __grid_constant__ RecoverArgs ra,
                          __nv_bfloat16 *__restrict__ act, __nv_bfloat16 *__restrict__ act_lo, DeviceStatus *status) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ float rscale_s[BM];
    __shared__ int acc_ok;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int c0 = (int)(blockIdx.x >> 1) * 2 * R, t0 = (int)rank * half, nt = min(B - t0, half);   // the pair's channels, this CTA's tokens
    const bool spare = c0 >= d_ff;   // the pair has no channels and recovers only
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const int wbytes = 2 * R * BK * 2, stage_bytes = kPairTokenBytes + wbytes, stages = gateup_pair_stages(R), kblocks = d / BK;
    Barriers *bars = reinterpret_cast<Barriers *>(base + stages * stage_bytes);
    if (threadIdx.x == 0) {
        prefetch_map(&tm_g); prefetch_map(&tm_u); prefetch_map(&tm_x); prefetch_map(&tm_x_lo);
        for (int s = 0; s < stages; ++s) { mbar_init(&bars->full[s], 1); mbar_init(&bars->empty[s], 1); }
        mbar_init(&bars->acc_ready, 1);
        bars->aborted = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1 && !spare) {   // the same warp of both CTAs allocates for the pair
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&bars->tmem_base)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();        // the peer's barriers exist before anything signals them
    tc_fence_after();

    if (spare && warp < kDecThreads / 32) {   // nothing to multiply
    } else if (warp == 0) {
        if (lane == 0) {
            const uint32_t full0 = map_to_cta(smem_u32(&bars->full[0]), 0);   // the even CTA's full barriers
            const int tx = 2 * (wbytes + 2 * half * BK * 2);                   // both CTAs' bytes
            const uint64_t once = policy_evict_first();
            auto load_w = [&](int kb, int s) {
                uint8_t *w = base + (size_t)s * stage_bytes + kPairTokenBytes;
                if (rank == 0) mbar_expect_tx(&bars->full[s], tx);
                tma_load_2d_pair(w, &tm_g, kb * BK, c0 + (int)rank * R, full0 + 8u * s, once);
                tma_load_2d_pair(w + wbytes / 2, &tm_u, kb * BK, c0 + (int)rank * R, full0 + 8u * s, once);
            };
            auto load_t = [&](int kb, int s) {
                uint8_t *t = base + (size_t)s * stage_bytes;
                tma_load_2d_pair(t, &tm_x, kb * BK, t0, full0 + 8u * s);
                tma_load_2d_pair(t + kABytes, &tm_x_lo, kb * BK, t0, full0 + 8u * s);
            };
            // weights are parameters: the first ring is requested before anything is waited for
            const int pre = min(stages, kblocks);
            for (int kb = 0; kb < pre; ++kb) load_w(kb, kb);
            pdl_wait();   // the token matrices
            for (int kb = 0; kb < pre; ++kb) load_t(kb, kb);
            int s = 0, ph = 0;
            for (int kb = pre; kb < kblocks; ++kb) {
                if (!mbar_wait(&bars->empty[s], ph, bars, status)) break;
                load_w(kb, s);
                load_t(kb, s);
                if (++s == stages) { s = 0; ph ^= 1; }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            // bf16 x bf16 -> f32, M = 256, N = 2 R
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * R >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
            const uint32_t tmem = bars->tmem_base;
            bool ok = true;
            int s = 0, ph = 0;
            for (int kb = 0; kb < kblocks; ++kb) {
                ok = mbar_wait(&bars->full[s], ph, bars, status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a0 = smem_u32(base + (size_t)s * stage_bytes), w0 = a0 + kPairTokenBytes;
#pragma unroll
                for (int k4 = 0; k4 < BK / 16; ++k4) {   // the descriptors' offsets hold in both CTAs' shared memory
                    const uint64_t hi = desc_sw128(a0 + k4 * 32, 16), lo = desc_sw128(a0 + kABytes + k4 * 32, 16);
                    const uint64_t g = desc_sw128(w0 + k4 * 32, 16), u = desc_sw128(w0 + wbytes / 2 + k4 * 32, 16);
                    tc_mma_pair(tmem, hi, g, idesc, (kb | k4) != 0);
                    tc_mma_pair(tmem, lo, g, idesc, 1);
                    tc_mma_pair(tmem + 256, hi, u, idesc, (kb | k4) != 0);
                    tc_mma_pair(tmem + 256, lo, u, idesc, 1);
                }
                tc_commit_pair(&bars->empty[s]);
                if (++s == stages) { s = 0; ph ^= 1; }
            }
            if (ok) tc_commit_pair(&bars->acc_ready);
        }
    } else if (warp < kDecThreads / 32) {
        const int et = threadIdx.x - 64, q = warp & 3, sub = (warp - 2) >> 2;
        pdl_wait();   // the row squares; and nothing is stored before the kernels before this one are complete
        for (int t = et; t < nt; t += kEpiThreads) {
            float rs = 1.f;
            if (ss_part != nullptr) {
                float sq = 0.f;
                for (int i = 0; i < d / 64; i += 16) {   // d is a multiple of 256
                    float v[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) v[u] = i + u < d / 64 ? ld_dep(ss_part + (size_t)(i + u) * B + t0 + t) : 0.f;
#pragma unroll
                    for (int u = 0; u < 16; ++u) sq += v[u];
                }
                rs = rsqrtf(sq / (float)d + eps);
            }
            rscale_s[t] = rs;
        }
        if (warp == 2) {   // one warp polls, the others sleep at the barrier behind it
            const bool ok = mbar_wait(&bars->acc_ready, 0, bars, status);
            if (lane == 0) acc_ok = ok;
        }
        epi_sync();
        tc_fence_after();
        // lane = token, eight channels at a time, two warps per lane quarter
        const int t = q * 32 + lane;
        const uint32_t tbase = bars->tmem_base + ((uint32_t)(q * 32) << 16);
        if (acc_ok && q * 32 < nt) {
            const float sc = t < nt ? rscale_s[t] : 0.f;
#pragma unroll 1
            for (int c = 8 * sub; c < 2 * R; c += 16) {
                uint32_t g[8], u[8];
                tc_ld8(tbase + c, g);
                tc_ld8(tbase + 256 + c, u);
                tc_wait_ld();
                if (t < nt && c0 + c < d_ff) {
                    float v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[j] = silu_f(__uint_as_float(g[j]) * sc) * (__uint_as_float(u[j]) * sc);
                    uint2 h0, l0, h1, l1;
                    split4(v[0], v[1], v[2], v[3], h0, l0);
                    split4(v[4], v[5], v[6], v[7], h1, l1);
                    const size_t off = (size_t)(t0 + t) * d_ff + c0 + c;
                    *reinterpret_cast<uint4 *>(act + off) = make_uint4(h0.x, h0.y, h1.x, h1.y);
                    *reinterpret_cast<uint4 *>(act_lo + off) = make_uint4(l0.x, l0.y, l1.x, l1.y);
                }
            }
        }
    } else {
        constexpr int kRecBar = 3;
        __shared__ RecoverSmem<kRecNW, KC> rs;
        const int g = threadIdx.x - kDecThreads;
        float phc[32];
        if (ra.m <= 32) recover_load_phi<kRecNW>(ra.Phi, ra.m, ra.G, g, phc);
        const GramSource M{ra.gram, gram_pitch(ra.G)};
        pdl_wait();   // the partial sketches and M come from the kernel before
        for (int t = blockIdx.x; t < B; t += gridDim.x) {
            recover_row<kRecNW, KC, kRecBar>(
                rs, ra, M, [&](auto &sm) { y_from_parts<kRecNW, kRecBar>(sm, ra.parts, g, t, ra.m); }, ra.mask, g, t, phc);
            bar_sync<kRecBar, kRecThreads>();
        }
        // this CTA's masks are written (the barrier that ends the loop, or no token at all)
        if (g == 0) {
            count_masks(ra.mask_count);
            pdl_launch_dependents();
        }
    }
    // Neither CTA leaves (or frees tensor memory) while the other may still read its shared memory or signal its barriers; every
    // wait above is bounded, so both reach this point.
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (warp == 1 && !spare) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(bars->tmem_base), "r"(512) : "memory");
    }
}

// ---- down -----------------------------------------------------------------------------------------------
// grid (d / 256, slices).  The list is every group (use_union == 0) or the groups that are in some token's support; slice z
// takes the 64-channel k blocks [z nk / Z, (z + 1) nk / Z) of it.  mask_count: the CTAs that have written their masks, all of them
// at mask_ctas (0: not counted).
template <bool PACK, int MT>
__global__ void __launch_bounds__(kDecThreads, 2)
decode_down_kernel(const __grid_constant__ CUtensorMap tm_wd, const __grid_constant__ CUtensorMap tm_act,
                   const __grid_constant__ CUtensorMap tm_act_lo, const int32_t *mask, const unsigned *mask_count,
                   unsigned mask_ctas, int use_union, int B, int G, int d, float *__restrict__ partial, DeviceStatus *status) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t union_s[4], masks_s;
    __shared__ int glist_s[kMaxG];                          // groups of this slice, in list order
    __shared__ __align__(16) uint32_t out_s[kMaxG][4 * MT]; // tokens whose support does not hold them: the lane masks
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const TokenTile tt = token_tile(PACK, MT, B);
    const int col0 = blockIdx.x * kDecBN, z = blockIdx.y, Z = gridDim.y;
    constexpr int wbytes = kDecBN * BK * 2;
    Barriers *bars = reinterpret_cast<Barriers *>(base + ring_bytes(tt, wbytes));
    const int stage_bytes = tt.bytes + wbytes;
    const int stages = ring_stages(tt, wbytes);
    const uint32_t tcols = MT == 2 ? 512u : 256u;
    pdl_launch_dependents();
    if (threadIdx.x == 0) { prefetch_map(&tm_wd); prefetch_map(&tm_act); prefetch_map(&tm_act_lo); }
    if (threadIdx.x < 4) union_s[threadIdx.x] = 0u;
    if (threadIdx.x == 64) {
        unsigned n = 0u;
        if (mask_ctas != 0u) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(n) : "l"(mask_count) : "memory");
        masks_s = mask_ctas != 0u && n == mask_ctas;
    }
    setup_cta(bars, warp, tcols);
    const bool masks_ready = masks_s != 0u;   // (behind a barrier, as the masks of the other threads' reads)
    if (use_union && !masks_ready) pdl_wait();
    int ng = G;
    if (use_union) {
        collect_union(mask, B, union_s);
        __syncthreads();
        ng = union_size(union_s);
    }
    const int nk = 2 * ng;
    const int k0 = (int)((long long)nk * z / Z), kblocks = (int)((long long)nk * (z + 1) / Z) - k0;
    const int l0 = k0 >> 1, nl = kblocks > 0 ? ((k0 + kblocks - 1) >> 1) - l0 + 1 : 0;   // list entries of this slice
    if (threadIdx.x < G) {
        const int g = threadIdx.x;
        int pos = g;
        bool in = true;
        if (use_union) {
            in = (union_s[g >> 5] >> (g & 31)) & 1u;
            pos = union_rank(union_s, g);
        }
        if (in && pos >= l0 && pos < l0 + nl) glist_s[pos - l0] = g;
    }
    __syncthreads();

    if (warp == 0) {
        if (lane == 0) {
            const int tx = wbytes + token_tx_bytes(tt);
            const uint64_t once = policy_evict_first();
            auto channel = [&](int kb) { return glist_s[((k0 + kb) >> 1) - l0] * 128 + ((k0 + kb) & 1) * BK; };
            auto load_w = [&](int ch, int s) {
                uint8_t *w = base + (size_t)s * stage_bytes + tt.bytes;
#pragma unroll
                for (int j = 0; j < kDecBN / 64; ++j)
                    tma_load_2d(w + j * (64 * BK * 2), &tm_wd, col0 + j * 64, ch, &bars->full[s], once);
            };
            const int pre = min(stages, kblocks);
            for (int kb = 0; kb < pre; ++kb) { mbar_expect_tx(&bars->full[kb], tx); load_w(channel(kb), kb); }
            pdl_wait();   // the activations
            for (int kb = 0; kb < pre; ++kb)
                load_tokens(tt, base + (size_t)kb * stage_bytes, &tm_act, &tm_act_lo, channel(kb), &bars->full[kb]);
            int s = 0, ph = 0;
            for (int kb = pre; kb < kblocks; ++kb) {
                if (!mbar_wait(&bars->empty[s], ph, bars, status)) break;
                mbar_expect_tx(&bars->full[s], tx);
                load_w(channel(kb), s);
                load_tokens(tt, base + (size_t)s * stage_bytes, &tm_act, &tm_act_lo, channel(kb), &bars->full[s]);
                if (++s == stages) { s = 0; ph ^= 1; }
            }
        }
    } else if (warp == 1) {
        asm volatile("bar.sync 2, %0;" ::"n"(kEpiThreads + 32) : "memory");   // accumulators zeroed, lane masks in place
        tc_fence_after();
        if (lane == 0 && kblocks > 0) {
            constexpr uint32_t idesc = make_idesc(true);
            const uint32_t tmem = bars->tmem_base;
            bool ok = true;
            int s = 0, ph = 0;
            for (int kb = 0; kb < kblocks; ++kb) {
                const uint4 *lanes = reinterpret_cast<const uint4 *>(out_s[((k0 + kb) >> 1) - l0]);
                ok = mbar_wait(&bars->full[s], ph, bars, status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a0 = smem_u32(base + (size_t)s * stage_bytes), w0 = a0 + tt.bytes;
                mma_kblock<PACK, MT>(tmem, a0, tt.lo_off, idesc, false,
                                     [&](int k4) { return desc_sw128(w0 + k4 * 2048, 64 * BK * 2); }, lanes);
                tc_commit(&bars->empty[s]);
                if (++s == stages) { s = 0; ph ^= 1; }
            }
            if (ok) tc_commit(&bars->acc_ready);
        }
    } else {
        const int ew = warp - 2, q = warp & 3, et = threadIdx.x - 64;
        for (int c = ew >> 2; c < MT * 256 / 16; c += kEpiWarps / 4)
            tc_st16_zero(bars->tmem_base + ((uint32_t)(q * 32) << 16) + c * 16);
        tc_wait_st();
        if (!masks_ready) pdl_wait();
        // lane masks: epilogue warp w holds the membership words of tokens 32 w .. 32 w + 31
        if (ew < (PACK ? 2 : 4 * MT)) {
            const int t = 32 * ew + lane;
            const uint4 m = t < B ? ld_l2(mask + (size_t)t * 4) : make_uint4(0u, 0u, 0u, 0u);
            for (int i = 0; i < nl; ++i) {
                const int g = glist_s[i], w = g >> 5;
                const uint32_t word = w == 0 ? m.x : w == 1 ? m.y : w == 2 ? m.z : m.w;
                const uint32_t out = ~__ballot_sync(0xffffffffu, (word >> (g & 31)) & 1u);
                if (lane == 0) {
                    out_s[i][ew] = out;
                    if (PACK) out_s[i][ew + 2] = out;   // the remainder rows of the same tokens
                }
            }
        }
        tc_fence_before();
        asm volatile("bar.sync 2, %0;" ::"n"(kEpiThreads + 32) : "memory");
        if (warp == 2 && kblocks > 0) mbar_wait(&bars->acc_ready, 0, bars, status);
        epi_sync();
        const bool ok = kblocks > 0 && *reinterpret_cast<volatile uint32_t *>(&bars->aborted) == 0u &&
                        mbar_wait(&bars->acc_ready, 0, bars, status);
        tc_fence_after();
        pdl_wait();   // nothing is stored before the kernels before this one are complete
        float *dump = reinterpret_cast<float *>(base);
        constexpr int P = kDecBN + 4;
#pragma unroll 1
        for (int t = 0; t < MT; ++t) {
            const int t0 = t * BM, rows = min(B - t0, PACK ? 64 : BM);
            if (t > 0) epi_sync();
            if (ok) dump_tile<PACK>(bars->tmem_base + t * 256, kDecBN / 16, dump, P, rows, warp, lane);
            epi_sync();
#pragma unroll 2
            for (int i = et; i < rows * (kDecBN / 4); i += kEpiThreads) {
                const int r = i / (kDecBN / 4), c = (i % (kDecBN / 4)) * 4;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);   // an empty slice contributes zero
                if (ok) v = row4<PACK>(dump, P, r, c);
                *reinterpret_cast<float4 *>(partial + ((size_t)z * B + t0 + r) * d + col0 + c) = v;
            }
        }
    }
    teardown_cta(bars, warp, tcols);
}

// out[t, :] = residual[t, :] + sum_z partial[z, t, :], slices added in index order, all loads of a thread in flight at once.
constexpr int kReduceThreads = 256;
__global__ void __launch_bounds__(kReduceThreads)
decode_reduce_kernel(const float *__restrict__ partial, int Z, int n4, const float *residual, float *out, unsigned *mask_count) {
    pdl_launch_dependents();
    const int i = blockIdx.x * kReduceThreads + threadIdx.x;
    pdl_wait();
    if (i == 0) *mask_count = 0u;
    if (i >= n4) return;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (residual != nullptr) s = ld_dep4(residual + 4 * (size_t)i);
    for (int z0 = 0; z0 < Z; z0 += 8) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            v[u] = z0 + u < Z ? ld_dep4(partial + 4 * ((size_t)(z0 + u) * n4 + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u) { s.x += v[u].x; s.y += v[u].y; s.z += v[u].z; s.w += v[u].w; }
    }
    reinterpret_cast<float4 *>(out)[i] = s;
}

// ---- given supports: operand split and membership masks (one CTA per token) --------------------------------
// check: validates the support row (ascending, distinct, in range).
constexpr int kPrepThreads = 256;
__global__ void __launch_bounds__(kPrepThreads)
decode_prep_kernel(const float *__restrict__ h, const int32_t *__restrict__ support, int d, int k, int G,
                   __nv_bfloat16 *__restrict__ x_hi, __nv_bfloat16 *__restrict__ x_lo, int32_t *__restrict__ mask, int check,
                   unsigned *mask_count, DeviceStatus *status) {
    __shared__ uint32_t m_s[4];
    const int t = blockIdx.x, tid = threadIdx.x;
    pdl_launch_dependents();
    if (tid < 4) m_s[tid] = 0u;
    __syncthreads();
    pdl_wait();
    if (tid < k) {
        const int g = ld_dep(support + (size_t)t * k + tid);
        const bool in = (unsigned)g < (unsigned)G;
        if (in) atomicOr(&m_s[g >> 5], 1u << (g & 31));
        if (check && (!in || (tid > 0 && ld_dep(support + (size_t)t * k + tid - 1) >= g)))
            atomicCAS(&status->code, 0, (int)CS_ERR_SUPPORT);
    }
    for (int c = tid; c < d / 4; c += kPrepThreads) {
        const float4 v = ld_dep4(h + (size_t)t * d + 4 * (size_t)c);
        uint2 hi, lo;
        split4(v.x, v.y, v.z, v.w, hi, lo);
        reinterpret_cast<uint2 *>(x_hi + (size_t)t * d)[c] = hi;
        reinterpret_cast<uint2 *>(x_lo + (size_t)t * d)[c] = lo;
    }
    __syncthreads();
    if (tid < 4) mask[(size_t)t * 4 + tid] = (int)m_s[tid];
    __syncthreads();
    if (tid == 0) count_masks(mask_count);
}

typedef void (*GateUpFn)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, int, int, int, int,
                         const int32_t *, const float *, float,
                         RecoverArgs, __nv_bfloat16 *, __nv_bfloat16 *, DeviceStatus *);
typedef void (*DownFn)(CUtensorMap, CUtensorMap, CUtensorMap, const int32_t *, const unsigned *, unsigned, int, int, int, int, float *,
                       DeviceStatus *);

// The recovery's list form in four lengths (24, 32, 56, 64 slots); 0: no recovery inside the launch.
int gateup_kc(const cs_plan *plan) { return plan->cfg.k <= 24 ? 3 : plan->cfg.k <= 32 ? 4 : plan->cfg.k <= 56 ? 7 : 8; }
template <bool PACK, int MT> GateUpFn gateup_fn_kc(int kc) {
    return kc == 0 ? decode_gateup_kernel<PACK, MT, 0> : kc == 3 ? decode_gateup_kernel<PACK, MT, 3>
         : kc == 4 ? decode_gateup_kernel<PACK, MT, 4> : kc == 7 ? decode_gateup_kernel<PACK, MT, 7>
         : decode_gateup_kernel<PACK, MT, 8>;
}
GateUpFn gateup_fn(int form, int kc) {   // form: 0 packed, 1 / 2 accumulators (2: given supports, or the recovery a launch ahead)
    return form == 0 ? gateup_fn_kc<true, 1>(kc) : form == 1 ? gateup_fn_kc<false, 1>(kc) : decode_gateup_kernel<false, 2, 0>;
}
typedef void (*GateUpPairFn)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, int, int, int, int, int, const float *, float, RecoverArgs,
                             __nv_bfloat16 *, __nv_bfloat16 *, DeviceStatus *);
GateUpPairFn gateup_pair_fn(int kc) {
    return kc == 3 ? decode_gateup_pair_kernel<3> : kc == 4 ? decode_gateup_pair_kernel<4> : kc == 7 ? decode_gateup_pair_kernel<7> : decode_gateup_pair_kernel<8>;
}
DownFn down_fn(int form) { return form == 0 ? decode_down_kernel<true, 1> : form == 1 ? decode_down_kernel<false, 1> : decode_down_kernel<false, 2>; }

}  // namespace

// Half of the most groups.  With k = 64 slots a recovery inside gate/up costs what one with 56 does (108 groups, k = 60: 3 tokens
// 72 to 75 us a step, 64 tokens 81 to 87; with the recovery as a launch of its own 89 and 95); a longer list does not fit the registers.
bool decode_recovers(const cs_plan *plan) { return plan->cfg.k <= 64; }

int decode_slices(const cs_plan *plan) {   // list slices of the down GEMM: one CTA per SM
    const int tiles = plan->cfg.d / kDecBN;
    return max(1, min(min(plan->sm_count / tiles, kDecMaxSlices), 2 * plan->G));
}

cs_status prepare_decode(cs_plan *plan) {
    CS_CUDA_TRY(plan, prefer_shared(decode_prep_kernel));
    CS_CUDA_TRY(plan, prefer_shared(decode_reduce_kernel));
    const int smem = 1024 + kDecRing + (int)sizeof(Barriers);
    CS_CUDA_TRY(plan, cudaFuncSetAttribute(gateup_pair_fn(gateup_kc(plan)), cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    for (int form = 0; form < 3; ++form) {
        CS_CUDA_TRY(plan, cudaFuncSetAttribute(gateup_fn(form, 0), cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        CS_CUDA_TRY(plan, cudaFuncSetAttribute(gateup_fn(form, gateup_kc(plan)), cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        CS_CUDA_TRY(plan, cudaFuncSetAttribute(down_fn(form), cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    }
    return CS_OK;
}

cs_status launch_decode_prep(cs_plan *plan, const float *h, const int32_t *support, int B, bool check, cudaStream_t st) {
    const cs_config &c = plan->cfg;
    __nv_bfloat16 *x_hi = static_cast<__nv_bfloat16 *>(plan->x_bf16);
    launch_pdl(true, decode_prep_kernel, dim3(B), dim3(kPrepThreads), 0, st, h, support, c.d, c.k, plan->G, x_hi,
               x_hi + (size_t)c.max_tokens * c.d, (int32_t *)plan->mask, check ? 1 : 0, plan->mask_count, plan->status);
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

cs_status launch_decode_ffn(cs_plan *plan, const cs_layer *L, int B, const RecoverArgs *recover, bool given, bool norm,
                            const float *residual, float *out, cudaStream_t st) {
    const cs_config &c = plan->cfg;
    const bool pack = B <= 64;
    const int mt = B <= BM ? 1 : 2, form = pack ? 0 : mt;
    const TokenTile tt = token_tile(pack, mt, B);
    const bool pair = recover != nullptr && mt == 2;
    const int unit = pair ? 16 : 8;   // the instructions take N = 2 R in units of 16, over a pair of CTAs of 32
    const int R = min(128, ((c.d_ff + plan->sm_count - 1) / plan->sm_count + unit - 1) & ~(unit - 1));
    int gateup_ctas = pair ? 2 * ((c.d_ff + 2 * R - 1) / (2 * R)) : (c.d_ff + R - 1) / R;
    // A pair's channels come in units of 32, so a narrow layer has few pairs, each with more tokens to recover in turn (8 groups of d = 256,
    // 200 tokens: 64 CTAs and four rounds of 3 us, where units of 8 had given 128 CTAs).  Pairs without channels take over where
    // that saves a round: that step 32.9 us, with the channels' pairs alone 46.6, on single CTAs 34.6; 24 groups of d = 1024, 256 tokens,
    // 43.1, 49.9, 44.5; 40 of d = 1024, 129 tokens, 37.4, 43.0, 42.2.
    if (pair) {
        const int rounds = (B + plan->sm_count - 1) / plan->sm_count;
        if (rounds < (B + gateup_ctas - 1) / gateup_ctas) gateup_ctas = max(gateup_ctas, ((B + rounds - 1) / rounds + 1) & ~1);
    }
    const int half = ((B + 1) / 2 + 7) & ~7;   // pair: tokens of the even CTA
    __nv_bfloat16 *x_hi = static_cast<__nv_bfloat16 *>(plan->x_bf16), *x_lo = x_hi + (size_t)c.max_tokens * c.d;
    __nv_bfloat16 *act = static_cast<__nv_bfloat16 *>(plan->act), *act_lo = act + (size_t)c.max_tokens * c.d_ff;
    // Given supports, more than 128 tokens: gate/up over the groups in use.  There a channel costs more than its bytes (7B, 200
    // tokens on the same 22 groups 82.7 us against 128.7, on 44 of the 86 93.2 against 127.6, on all of them 129.4 against 129.5).  Up to 128 tokens
    // the weights requested ahead of the masks are worth as much as the groups left out (5 to 20 tokens on the same quarter
    // of the groups 42 to 46 us either way; on independent supports 47 to 54 with every group, 55 to 64 by the list).
    const bool by_list = given && mt == 2;
    CUtensorMap tm_g, tm_u, tm_gu = {}, tm_uu = {}, tm_x, tm_x_lo, tm_wd, tm_act, tm_act_lo;
    if (!make_map(&tm_g, L->W_gate, c.d, c.d_ff, c.d, R) || !make_map(&tm_u, L->W_up, c.d, c.d_ff, c.d, R) ||
        (by_list && (!make_map(&tm_gu, L->W_gate, c.d, c.d_ff, c.d, kListRows) || !make_map(&tm_uu, L->W_up, c.d, c.d_ff, c.d, kListRows))) ||
        !make_map(&tm_x, x_hi, c.d, B, c.d, tt.box) || !make_map(&tm_x_lo, x_lo, c.d, B, c.d, tt.box) ||
        !make_map(&tm_wd, L->Wd_t, c.d, c.d_ff, c.d, BK) || !make_map(&tm_act, act, c.d_ff, B, c.d_ff, tt.box) ||
        !make_map(&tm_act_lo, act_lo, c.d_ff, B, c.d_ff, tt.box))
        return record_cuda(plan, cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    {
        StageTimer timer(plan, CS_STAGE_EXEC, st);
        if (recover != nullptr) plan->stage_seen[CS_STAGE_RECOVER] = 0;   // part of this launch
        if (pair) {
            CUtensorMap tm_h, tm_h_lo;
            if (!make_map(&tm_h, x_hi, c.d, B, c.d, half) || !make_map(&tm_h_lo, x_lo, c.d, B, c.d, half))
                return record_cuda(plan, cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
            launch_pdl(true, gateup_pair_fn(gateup_kc(plan)), dim3(gateup_ctas), dim3(kDecThreads + kRecThreads),
                       1024 + (size_t)gateup_pair_stages(R) * (kPairTokenBytes + 2 * R * BK * 2) + sizeof(Barriers), st, tm_h, tm_h_lo, tm_g, tm_u, B, half,
                       R, c.d, c.d_ff, norm ? (const float *)sketch_square_partials(plan, B) : (const float *)nullptr, c.rms_eps, *recover, act,
                       act_lo, plan->status);
        } else {
            launch_pdl(true, gateup_fn(form, recover != nullptr ? gateup_kc(plan) : 0), dim3(gateup_ctas),
                       dim3(kDecThreads + (recover != nullptr ? kRecThreads : 0)),
                       by_list ? 1024 + (size_t)kDecRing + sizeof(Barriers) : decode_smem(tt, 2 * R * BK * 2), st, tm_x, tm_x_lo, tm_g, tm_u, tm_gu,
                       tm_uu, B, R, c.d, c.d_ff, by_list ? (const int32_t *)plan->mask : (const int32_t *)nullptr,
                       norm ? (const float *)sketch_square_partials(plan, B) : (const float *)nullptr, c.rms_eps,
                       recover != nullptr ? *recover : RecoverArgs{}, act, act_lo, plan->status);
        }
        plan->launches++;
        CS_CUDA_TRY(plan, cudaGetLastError());
    }
    const int Z = decode_slices(plan);
    {
        StageTimer timer(plan, CS_STAGE_EXEC2, st);
        // Expected number of groups in nobody's support, G (1 - k/G)^B: below a quarter group the list is every group and
        // need not be made.  (7B, 5 tokens, 19.6 groups expected: 48.4 us with the union, 52.1 with every group; 8 tokens, 8.1: 51.8
        // and 53.2; from 11 tokens, 3.3 groups, on the two are equal within the spread, so the line is not critical.)
        const bool use_union = by_list || (float)plan->G * powf(1.f - (float)c.k / plan->G, (float)B) > 0.25f;
        launch_pdl(true, down_fn(form), dim3(c.d / kDecBN, Z), dim3(kDecThreads), decode_smem(tt, kDecBN * BK * 2), st, tm_wd, tm_act,
                   tm_act_lo, (const int32_t *)plan->mask, (const unsigned *)plan->mask_count,
                   recover != nullptr ? (unsigned)gateup_ctas : given ? (unsigned)B : 0u, use_union ? 1 : 0, B, plan->G, c.d, plan->mma_partial, plan->status);
        plan->launches++;
        CS_CUDA_TRY(plan, cudaGetLastError());
    }
    {
        StageTimer timer(plan, CS_STAGE_REDUCE, st);
        const int n4 = B * c.d / 4;
        launch_pdl(true, decode_reduce_kernel, dim3((n4 + kReduceThreads - 1) / kReduceThreads), dim3(kReduceThreads), 0, st,
                   (const float *)plan->mma_partial, Z, n4, residual, out, plan->mask_count);
        plan->launches++;
        CS_CUDA_TRY(plan, cudaGetLastError());
    }
    return CS_OK;
}

}  // namespace cs
