// Actuator, tensor-core regime for decode batches of at most kDecodeMaxTokens tokens with independent supports.
//
//   decode_gateup_kernel   act[t, c] = silu(n_t . W_gate[c]) (n_t . W_up[c]) for every channel c, zero where the
//                          channel's group is not in the token's support
//   decode_down_kernel     partial[z, t, :] = sum over the channels of list slice z of act[t, c] Wd_t[c, :]
//   reduce_slices_kernel   out = residual + sum_z partial
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
// columns; MT = 2 (more than 128 tokens) keeps two accumulators.  Rows no token owns hold whatever shared memory
// held: rows of an MMA do not mix, and those results are never read.
//
// Balance: the channel tiles of gate/up are not tied to the 128-channel groups.  A CTA takes R channels, R the
// multiple of 8 that gives every SM one CTA (80 at d_ff = 11008: 138 CTAs on 148 SMs; one CTA per group left 62 SMs
// without work and took 39.7 us for 180 MB at 64 tokens).  The down GEMM has d / 256 column tiles times
// as many list slices as fill the SMs, cut at 64-channel k blocks.
//
// Chain: gate/up does not need the supports until its epilogue.  In a step the launch before it is the recovery,
// which triggers its programmatic dependents as soon as the kernels before IT have completed; gate/up then streams
// while the recovery runs beside it on the same SMs and waits for it (griddepcontrol.wait) only when the accumulators
// are complete.  The down kernel requests its first ring of weights before it waits for the activations.
#include "mma_core.cuh"

namespace cs {

namespace {

constexpr int kEpiWarps = 8;                         // two per quarter of the tensor-memory lanes
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kDecThreads = 64 + kEpiThreads;        // + TMA warp, MMA warp
constexpr int kDecRing = 208 * 1024;                 // operand ring; what is left of the 227 KB holds the recovery's CTAs
constexpr size_t kDecSmem = 1024 + (size_t)kDecRing + 256;
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
__device__ __forceinline__ int ring_stages(const TokenTile &t, int wbytes) {
    return min(kMaxStages, (kDecRing - max(0, t.over - wbytes)) / (t.bytes + wbytes));
}
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
template <bool PACK, int MT, typename BDesc>
__device__ __forceinline__ void mma_kblock(uint32_t tmem, uint32_t a0, uint32_t lo_off, uint32_t idesc, bool first, BDesc bdesc) {
#pragma unroll
    for (int k4 = 0; k4 < BK / 16; ++k4) {
        const uint64_t bd = bdesc(k4);
#pragma unroll
        for (int t = 0; t < MT; ++t) {
            const uint32_t a = a0 + t * kABytes + k4 * 32;
            tc_mma(tmem + t * 256, desc_sw128(a, 16), bd, idesc, !first || k4 != 0);
            if (!PACK) tc_mma(tmem + t * 256, desc_sw128(a + lo_off, 16), bd, idesc, 1);
        }
    }
}

// ---- gate / up ------------------------------------------------------------------------------------------
// CTA x: channels [x R, x R + R).  x_ready: the token matrices were complete before this launch could begin.
template <bool PACK, int MT>
__global__ void __launch_bounds__(kDecThreads, 2)
decode_gateup_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_x_lo,
                     const __grid_constant__ CUtensorMap tm_g, const __grid_constant__ CUtensorMap tm_u, int B, int R, int d,
                     int d_ff, int x_ready, const int32_t *mask, const float *rscale,
                     __nv_bfloat16 *__restrict__ act, __nv_bfloat16 *__restrict__ act_lo, DeviceStatus *status) {
    extern __shared__ uint8_t smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    Barriers *bars = reinterpret_cast<Barriers *>(base + kDecRing);
    const TokenTile tt = token_tile(PACK, MT, B);
    const int c0 = blockIdx.x * R;
    const int wbytes = 2 * R * BK * 2;                   // gate rows then up rows
    const int stage_bytes = tt.bytes + wbytes;
    const int stages = ring_stages(tt, wbytes);
    const uint32_t tcols = MT == 2 ? 512u : 256u;
    const int kblocks = d / BK;
    if (threadIdx.x == 0) { prefetch_map(&tm_g); prefetch_map(&tm_u); prefetch_map(&tm_x); prefetch_map(&tm_x_lo); }
    setup_cta(bars, warp, tcols);

    if (warp == 0) {
        if (lane == 0) {
            const int tx = wbytes + token_tx_bytes(tt);
            auto load_w = [&](int kb, int s) {
                uint8_t *w = base + (size_t)s * stage_bytes + tt.bytes;
                tma_load_2d(w, &tm_g, kb * BK, c0, &bars->full[s]);
                tma_load_2d(w + wbytes / 2, &tm_u, kb * BK, c0, &bars->full[s]);
            };
            // weights are parameters: the first ring is requested before anything is waited for
            const int pre = min(stages, kblocks);
            for (int kb = 0; kb < pre; ++kb) { mbar_expect_tx(&bars->full[kb], tx); load_w(kb, kb); }
            if (!x_ready) pdl_wait();
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
    } else {
        const bool ok = mbar_wait(&bars->acc_ready, 0, bars, status);
        tc_fence_after();
        pdl_wait();                  // the supports (and the row scales) are final
        pdl_launch_dependents();     // the down kernel reads the supports before its own wait
        float *dump = reinterpret_cast<float *>(base);   // the ring is free: every load has been consumed
        const int P = ((2 * R + 31) & ~31) + 4;
        const int et = threadIdx.x - 64, r4 = R / 4;
#pragma unroll 1
        for (int t = 0; t < MT; ++t) {
            const int t0 = t * BM, rows = min(B - t0, PACK ? 64 : BM);
            if (t > 0) epi_sync();
            if (ok) dump_tile<PACK>(bars->tmem_base + t * 256, 2 * R / 16, dump, P, rows, warp, lane);
            epi_sync();
            if (ok) {
                for (int i = et; i < rows * r4; i += kEpiThreads) {
                    const int r = i / r4, c = (i - r * r4) * 4, ch = c0 + c;
                    if (ch >= d_ff) continue;
                    const float4 g = row4<PACK>(dump, P, r, c), u = row4<PACK>(dump, P, r, R + c);
                    const int grp = ch >> 7;
                    const bool in = ((uint32_t)ld_dep(mask + (size_t)(t0 + r) * 4 + (grp >> 5)) >> (grp & 31)) & 1u;
                    float a[4] = {0.f, 0.f, 0.f, 0.f};
                    if (in) {
                        const float sc = rscale != nullptr ? ld_dep(rscale + t0 + r) : 1.f;
                        a[0] = silu_f(g.x * sc) * (u.x * sc); a[1] = silu_f(g.y * sc) * (u.y * sc);
                        a[2] = silu_f(g.z * sc) * (u.z * sc); a[3] = silu_f(g.w * sc) * (u.w * sc);
                    }
                    uint2 hi, lo;
                    split4(a[0], a[1], a[2], a[3], hi, lo);
                    const size_t off = (size_t)(t0 + r) * d_ff + ch;
                    *reinterpret_cast<uint2 *>(act + off) = hi;
                    *reinterpret_cast<uint2 *>(act_lo + off) = lo;
                }
            }
        }
    }
    teardown_cta(bars, warp, tcols);
}

// ---- down -----------------------------------------------------------------------------------------------
// grid (d / 256, slices).  The list is every group (use_union == 0) or the groups that are in some token's support; slice z
// takes the 64-channel k blocks [z nk / Z, (z + 1) nk / Z) of it.
template <bool PACK, int MT>
__global__ void __launch_bounds__(kDecThreads, 2)
decode_down_kernel(const __grid_constant__ CUtensorMap tm_wd, const __grid_constant__ CUtensorMap tm_act,
                   const __grid_constant__ CUtensorMap tm_act_lo, const int32_t *mask, int use_union, int B, int G,
                   int d, float *__restrict__ partial, DeviceStatus *status) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint32_t union_s[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    Barriers *bars = reinterpret_cast<Barriers *>(base + kDecRing);
    const TokenTile tt = token_tile(PACK, MT, B);
    const int col0 = blockIdx.x * kDecBN, z = blockIdx.y, Z = gridDim.y;
    constexpr int wbytes = kDecBN * BK * 2;
    const int stage_bytes = tt.bytes + wbytes;
    const int stages = ring_stages(tt, wbytes);
    const uint32_t tcols = MT == 2 ? 512u : 256u;
    pdl_launch_dependents();
    if (threadIdx.x == 0) { prefetch_map(&tm_wd); prefetch_map(&tm_act); prefetch_map(&tm_act_lo); }
    if (threadIdx.x < 4) union_s[threadIdx.x] = 0u;
    setup_cta(bars, warp, tcols);
    int ng = G;
    if (use_union) {   // the supports were final before this launch could begin (see the gate/up kernel's trigger)
        for (int t = threadIdx.x; t < B; t += kDecThreads) {
            const uint4 m = ld_l2(mask + (size_t)t * 4);
            if (m.x) atomicOr(&union_s[0], m.x);
            if (m.y) atomicOr(&union_s[1], m.y);
            if (m.z) atomicOr(&union_s[2], m.z);
            if (m.w) atomicOr(&union_s[3], m.w);
        }
        __syncthreads();
        ng = __popc(union_s[0]) + __popc(union_s[1]) + __popc(union_s[2]) + __popc(union_s[3]);
    }
    const int nk = 2 * ng;
    const int k0 = (int)((long long)nk * z / Z), kblocks = (int)((long long)nk * (z + 1) / Z) - k0;

    if (warp == 0) {
        if (lane == 0) {
            const int tx = wbytes + token_tx_bytes(tt);
            // walks the channels of the list's k blocks: two per group
            struct Walk { int word; uint32_t bits; int g; bool half; };
            auto start = [&](int k) {
                Walk w{0, 0u, k >> 1, (k & 1) != 0};
                if (use_union) {
                    int skip = k >> 1;
                    while (w.word < 3 && skip >= __popc(union_s[w.word])) skip -= __popc(union_s[w.word++]);
                    w.bits = union_s[w.word];
                    while (skip-- > 0) w.bits &= w.bits - 1;
                    w.g = 32 * w.word + __ffs(w.bits) - 1;
                }
                return w;
            };
            auto channel = [](const Walk &w) { return w.g * 128 + (w.half ? BK : 0); };
            auto advance = [&](Walk &w) {
                if (!w.half) { w.half = true; return; }
                w.half = false;
                if (!use_union) { ++w.g; return; }
                w.bits &= w.bits - 1;
                while (w.bits == 0u && w.word < 3) w.bits = union_s[++w.word];
                w.g = 32 * w.word + __ffs(w.bits) - 1;
            };
            auto load_w = [&](int ch, int s) {
                uint8_t *w = base + (size_t)s * stage_bytes + tt.bytes;
#pragma unroll
                for (int j = 0; j < kDecBN / 64; ++j)
                    tma_load_2d(w + j * (64 * BK * 2), &tm_wd, col0 + j * 64, ch, &bars->full[s]);
            };
            const int pre = min(stages, kblocks);
            if (kblocks > 0) {
                Walk w = start(k0), wa = w;
                for (int kb = 0; kb < pre; ++kb, advance(w)) { mbar_expect_tx(&bars->full[kb], tx); load_w(channel(w), kb); }
                pdl_wait();   // the activations
                for (int kb = 0; kb < pre; ++kb, advance(wa))
                    load_tokens(tt, base + (size_t)kb * stage_bytes, &tm_act, &tm_act_lo, channel(wa), &bars->full[kb]);
                int s = 0, ph = 0;
                for (int kb = pre; kb < kblocks; ++kb, advance(w)) {
                    if (!mbar_wait(&bars->empty[s], ph, bars, status)) break;
                    mbar_expect_tx(&bars->full[s], tx);
                    load_w(channel(w), s);
                    load_tokens(tt, base + (size_t)s * stage_bytes, &tm_act, &tm_act_lo, channel(w), &bars->full[s]);
                    if (++s == stages) { s = 0; ph ^= 1; }
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && kblocks > 0) {
            constexpr uint32_t idesc = make_idesc(true);
            const uint32_t tmem = bars->tmem_base;
            bool ok = true;
            int s = 0, ph = 0;
            for (int kb = 0; kb < kblocks; ++kb) {
                ok = mbar_wait(&bars->full[s], ph, bars, status);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a0 = smem_u32(base + (size_t)s * stage_bytes), w0 = a0 + tt.bytes;
                mma_kblock<PACK, MT>(tmem, a0, tt.lo_off, idesc, kb == 0,
                                     [&](int k4) { return desc_sw128(w0 + k4 * 2048, 64 * BK * 2); });
                tc_commit(&bars->empty[s]);
                if (++s == stages) { s = 0; ph ^= 1; }
            }
            if (ok) tc_commit(&bars->acc_ready);
        }
    } else {
        const bool ok = kblocks > 0 && mbar_wait(&bars->acc_ready, 0, bars, status);
        tc_fence_after();
        pdl_wait();   // nothing is stored before the kernels before this one are complete
        float *dump = reinterpret_cast<float *>(base);
        constexpr int P = kDecBN + 4;
        const int et = threadIdx.x - 64;
#pragma unroll 1
        for (int t = 0; t < MT; ++t) {
            const int t0 = t * BM, rows = min(B - t0, PACK ? 64 : BM);
            if (t > 0) epi_sync();
            if (ok) dump_tile<PACK>(bars->tmem_base + t * 256, kDecBN / 16, dump, P, rows, warp, lane);
            epi_sync();
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
decode_reduce_kernel(const float *__restrict__ partial, int Z, int n4, const float *residual, float *out) {
    pdl_launch_dependents();
    const int i = blockIdx.x * kReduceThreads + threadIdx.x;
    pdl_wait();
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
// check: validates the support row (ascending, distinct, in range).  x_hi == NULL: masks only.
constexpr int kPrepThreads = 256;
__global__ void __launch_bounds__(kPrepThreads)
decode_prep_kernel(const float *__restrict__ h, const int32_t *__restrict__ support, int d, int k, int G,
                   __nv_bfloat16 *__restrict__ x_hi, __nv_bfloat16 *__restrict__ x_lo, int32_t *__restrict__ mask, int check,
                   DeviceStatus *status) {
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
    if (x_hi != nullptr) {
        for (int c = tid; c < d / 4; c += kPrepThreads) {
            const float4 v = ld_dep4(h + (size_t)t * d + 4 * (size_t)c);
            uint2 hi, lo;
            split4(v.x, v.y, v.z, v.w, hi, lo);
            reinterpret_cast<uint2 *>(x_hi + (size_t)t * d)[c] = hi;
            reinterpret_cast<uint2 *>(x_lo + (size_t)t * d)[c] = lo;
        }
    }
    __syncthreads();
    if (tid < 4) mask[(size_t)t * 4 + tid] = (int)m_s[tid];
}

typedef void (*GateUpFn)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, int, int, int, int, int, const int32_t *,
                         const float *, __nv_bfloat16 *, __nv_bfloat16 *, DeviceStatus *);
typedef void (*DownFn)(CUtensorMap, CUtensorMap, CUtensorMap, const int32_t *, int, int, int, int, float *, DeviceStatus *);

}  // namespace

int decode_slices(const cs_plan *plan) {   // list slices of the down GEMM: one CTA per SM
    const int tiles = plan->cfg.d / kDecBN;
    return max(1, min(min(plan->sm_count / tiles, kDecMaxSlices), 2 * plan->G));
}

cs_status prepare_decode(cs_plan *plan) {
    CS_CUDA_TRY(plan, prefer_shared(decode_prep_kernel));
    CS_CUDA_TRY(plan, prefer_shared(decode_reduce_kernel));
    const int smem = (int)kDecSmem;
    CS_CUDA_TRY(plan, cudaFuncSetAttribute(decode_gateup_kernel<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CS_CUDA_TRY(plan, cudaFuncSetAttribute(decode_gateup_kernel<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CS_CUDA_TRY(plan, cudaFuncSetAttribute(decode_gateup_kernel<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CS_CUDA_TRY(plan, cudaFuncSetAttribute(decode_down_kernel<true, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CS_CUDA_TRY(plan, cudaFuncSetAttribute(decode_down_kernel<false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    CS_CUDA_TRY(plan, cudaFuncSetAttribute(decode_down_kernel<false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return CS_OK;
}

cs_status launch_decode_prep(cs_plan *plan, const float *h, const int32_t *support, int B, bool check, cudaStream_t st) {
    const cs_config &c = plan->cfg;
    __nv_bfloat16 *x_hi = static_cast<__nv_bfloat16 *>(plan->x_bf16);
    launch_pdl(true, decode_prep_kernel, dim3(B), dim3(kPrepThreads), 0, st, h, support, c.d, c.k, plan->G, h ? x_hi : nullptr,
               x_hi + (size_t)c.max_tokens * c.d, (int32_t *)plan->mask, check ? 1 : 0, plan->status);
    plan->launches++;
    CS_CUDA_TRY(plan, cudaGetLastError());
    return CS_OK;
}

// The three launches of the actuator.  The token matrices (plan->x_bf16), the masks (plan->mask) and, with rscale, the row
// scales (plan->rscale) come from the launches before; x_ready: the launch directly before this one triggers its
// dependents only after the matrices are complete.
cs_status launch_decode_ffn(cs_plan *plan, const cs_layer *L, int B, bool x_ready, bool rscale, const float *residual, float *out,
                            cudaStream_t st) {
    const cs_config &c = plan->cfg;
    const bool pack = B <= 64;
    const int mt = B <= BM ? 1 : 2;
    const TokenTile tt = token_tile(pack, mt, B);
    const int R = min(128, ((c.d_ff + plan->sm_count - 1) / plan->sm_count + 7) & ~7);
    __nv_bfloat16 *x_hi = static_cast<__nv_bfloat16 *>(plan->x_bf16), *x_lo = x_hi + (size_t)c.max_tokens * c.d;
    __nv_bfloat16 *act = static_cast<__nv_bfloat16 *>(plan->act), *act_lo = act + (size_t)c.max_tokens * c.d_ff;
    CUtensorMap tm_g, tm_u, tm_x, tm_x_lo, tm_wd, tm_act, tm_act_lo;
    if (!make_map(&tm_g, L->W_gate, c.d, c.d_ff, c.d, R) || !make_map(&tm_u, L->W_up, c.d, c.d_ff, c.d, R) ||
        !make_map(&tm_x, x_hi, c.d, B, c.d, tt.box) || !make_map(&tm_x_lo, x_lo, c.d, B, c.d, tt.box) ||
        !make_map(&tm_wd, L->Wd_t, c.d, c.d_ff, c.d, BK) || !make_map(&tm_act, act, c.d_ff, B, c.d_ff, tt.box) ||
        !make_map(&tm_act_lo, act_lo, c.d_ff, B, c.d_ff, tt.box))
        return record_cuda(plan, cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
    {
        StageTimer timer(plan, CS_STAGE_EXEC, st);
        const GateUpFn fn = pack ? decode_gateup_kernel<true, 1> : mt == 1 ? decode_gateup_kernel<false, 1> : decode_gateup_kernel<false, 2>;
        launch_pdl(true, fn, dim3((c.d_ff + R - 1) / R), dim3(kDecThreads), kDecSmem, st, tm_x, tm_x_lo, tm_g, tm_u, B, R, c.d, c.d_ff,
                   x_ready ? 1 : 0, (const int32_t *)plan->mask, rscale ? (const float *)plan->rscale : (const float *)nullptr, act, act_lo,
                   plan->status);
        plan->launches++;
        CS_CUDA_TRY(plan, cudaGetLastError());
    }
    const int Z = decode_slices(plan);
    {
        StageTimer timer(plan, CS_STAGE_EXEC2, st);
        // Expected number of groups in nobody's support, G (1 - k/G)^B: below a quarter group the list is every group and
        // the masks need not be read.
        const bool use_union = (float)plan->G * powf(1.f - (float)c.k / plan->G, (float)B) > 0.25f;
        const DownFn fn = pack ? decode_down_kernel<true, 1> : mt == 1 ? decode_down_kernel<false, 1> : decode_down_kernel<false, 2>;
        launch_pdl(true, fn, dim3(c.d / kDecBN, Z), dim3(kDecThreads), kDecSmem, st, tm_wd, tm_act, tm_act_lo, (const int32_t *)plan->mask,
                   use_union ? 1 : 0, B, plan->G, c.d, plan->mma_partial, plan->status);
        plan->launches++;
        CS_CUDA_TRY(plan, cudaGetLastError());
    }
    {
        StageTimer timer(plan, CS_STAGE_REDUCE, st);
        const int n4 = B * c.d / 4;
        launch_pdl(true, decode_reduce_kernel, dim3((n4 + kReduceThreads - 1) / kReduceThreads), dim3(kReduceThreads), 0, st,
                   (const float *)plan->mma_partial, Z, n4, residual, out);
        plan->launches++;
        CS_CUDA_TRY(plan, cudaGetLastError());
    }
    return CS_OK;
}

}  // namespace cs
