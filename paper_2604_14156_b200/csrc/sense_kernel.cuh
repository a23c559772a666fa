// Sensor and estimator of a token in one launch (small batches, the prompt's mean).
// A cluster of eight CTAs per token.  CTA r takes the columns [r d / 8, (r + 1) d / 8) of S and x.  Its part of S is in
// shared memory before the wait for the kernel that produces x, and so are Phi and M = I - mu Phi^T Phi in that of
// CTA 0 (every CTA forms an eighth of M), so between x and the sketch lie one load of x, the dot products, and one
// exchange over distributed shared memory; CTA 0 then runs the iteration with every operand in its shared memory.
// Bound by latency.  As two launches, with M formed by the first and read from L2 by the second, the pair took
// 15 us of a step at 7B, batch 1 (to the gather kernel), in this form 10 us (26.1 us for the step against 29.8).
#pragma once
#include "sense.cuh"

namespace cs {

__device__ __forceinline__ uint32_t remote_smem(const void *p, uint32_t rank) {   // the same place in CTA `rank` of the cluster
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_remote(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// STAGED: x is a prompt's column sums, which every CTA adds up once for all its warps.
// PLAIN: see recover_row.  NORM: without an RMSNorm, with one, or either (2).  ALL: every row of S has its place in shared memory.
// What is bound by latency here is also the fetch of code that the weights of the step before have pushed out of the caches around
// the SMs: what a form never runs is left out of it, so that what it runs lies close together.  One kernel for all of them, and
// now: 7B, one token 25.6 and 24.6 us a step, three 41.8 and 39.3; 8B, four 58.3 and 54.9; 777 prompt tokens 72.9 and 69.7.
template <int NW, int KC, bool STAGED, bool PLAIN, int NORM, bool ALL>
__global__ void __cluster_dims__(kSenseCtas, 1, 1) __launch_bounds__(kSenseThreads, 1)
sense_recover_kernel(const __grid_constant__ SenseArgs sa, const __grid_constant__ RecoverArgs a) {
    constexpr int GP = 32 * NW;
    const bool norm = NORM == 2 ? sa.gamma != nullptr : NORM == 1;
    extern __shared__ float4 sense_s[];
    __shared__ RecoverSmem<NW, KC> rs;
    __shared__ float part_s[kSenseCtas][kMaxM], ss_s[kSenseCtas];
    const int t = blockIdx.x / kSenseCtas, rank = blockIdx.x % kSenseCtas;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m = a.m, G = a.G, d = sa.d;
    const int nc = d / (4 * kSenseCtas);            // float4 columns of this CTA
    const size_t col0 = (size_t)rank * nc * 4;
    const int pitch = (G + 3) & ~3, ppitch = pitch + 4;
    float *M_s = reinterpret_cast<float *>(sense_s), *phi_s = M_s + G * pitch;
    float4 *S_s = reinterpret_cast<float4 *>(phi_s + m * ppitch);
    pdl_launch_dependents();
    cluster_arrive();                               // matched below: every CTA of the cluster has started
    // this lane's chunks of this warp's rows of S (read by this warp only)
    for (int r = warp; r < sa.s_rows; r += kSenseWarps)
#pragma unroll 4
        for (int c = lane; c < nc; c += 32) {
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(S_s + r * nc + c);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(sa.S + (size_t)r * d + col0 + 4 * c) : "memory");
        }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int nch = (nc + 31) / 32;
    // rows of S without a place there: the warp's next in registers, what is left in L2 at least
    float4 ex[kSenseExtra][kSenseMaxChunks];
    const int x0 = sa.s_rows + ((warp - sa.s_rows) & (kSenseWarps - 1));   // this warp's first such row
    if constexpr (!ALL) {
#pragma unroll
        for (int q = 0; q < kSenseExtra; ++q)
#pragma unroll
            for (int j = 0; j < kSenseMaxChunks; ++j)
                if (x0 + q * kSenseWarps < m && j < nch)
                    ex[q][j] = __ldg(reinterpret_cast<const float4 *>(sa.S + (size_t)(x0 + q * kSenseWarps) * d + col0) + min(lane + 32 * j, nc - 1));
        for (int r = sa.s_rows + kSenseExtra * kSenseWarps + tid; r < m; r += kSenseThreads)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(sa.S + (size_t)r * d + col0), "r"(nc * 16) : "memory");
    }
    for (int i0 = tid; i0 < m * GP; i0 += 8 * kSenseThreads) {   // eight loads in flight: addresses clamped, no branches
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = min(i0 + u * kSenseThreads, m * GP - 1);
            v[u] = __ldg(a.Phi + i / GP * G + min(i % GP, G - 1));
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int i = i0 + u * kSenseThreads, g = i % GP;
            if (i < m * GP && g < pitch) phi_s[i / GP * ppitch + g] = g < G ? v[u] : 0.f;
        }
    }
    __syncthreads();
    float phc[32];
    if (rank == 0 && tid < GP) recover_init<!PLAIN>(rs, tid, m, a.k);
    if (rank == 0 && m <= 32 && tid < GP) {
#pragma unroll
        for (int row = 0; row < 32; ++row) phc[row] = row < m && tid < G ? phi_s[row * ppitch + tid] : 0.f;
    }
    cluster_wait();
    // M in blocks of 2 x 4 entries, each summed as gram_rows sums it; every eighth row pair is this CTA's
    const uint32_t M0 = remote_smem(M_s, 0);
    for (int b = tid; b < ((G + 1) / 2 - rank + kSenseCtas - 1) / kSenseCtas * (pitch / 4); b += kSenseThreads) {
        const int i0 = (b / (pitch / 4) * kSenseCtas + rank) * 2, j0 = b % (pitch / 4) * 4;
        float s0[2][4] = {}, s1[2][4] = {};
        auto add = [&](int row, float (&s)[2][4]) {
            const float2 p = *reinterpret_cast<const float2 *>(phi_s + row * ppitch + i0);
            const float4 q = *reinterpret_cast<const float4 *>(phi_s + row * ppitch + j0);
            s[0][0] = fmaf(p.x, q.x, s[0][0]); s[0][1] = fmaf(p.x, q.y, s[0][1]); s[0][2] = fmaf(p.x, q.z, s[0][2]); s[0][3] = fmaf(p.x, q.w, s[0][3]);
            s[1][0] = fmaf(p.y, q.x, s[1][0]); s[1][1] = fmaf(p.y, q.y, s[1][1]); s[1][2] = fmaf(p.y, q.z, s[1][2]); s[1][3] = fmaf(p.y, q.w, s[1][3]);
        };
        int row = 0;
#pragma unroll 4
        for (; row + 1 < m; row += 2) { add(row, s0); add(row + 1, s1); }
        if (row < m) add(row, s0);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (i0 + u >= G) break;
            float o[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) o[v] = j0 + v < G ? (i0 + u == j0 + v ? 1.f : 0.f) - a.mu * (s0[u][v] + s1[u][v]) : 0.f;
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(M0 + 4u * ((i0 + u) * pitch + j0)), "f"(o[0]), "f"(o[1]),
                         "f"(o[2]), "f"(o[3]) : "memory");
        }
    }
    // A lane's wait covers its own copies; when nc is not a multiple of 32 the lanes past the end read the last column, which
    // another lane copied (their x is zero, but zero times what shared memory held before could be NaN).
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    pdl_wait();   // x may be the previous kernel's output
    float4 xv[kSenseMaxChunks], gm[kSenseMaxChunks];
    float ss = 0.f;
    if (norm) {
#pragma unroll
        for (int j = 0; j < kSenseMaxChunks; ++j)
            if (j < nch) gm[j] = __ldg(reinterpret_cast<const float4 *>(sa.gamma + col0) + min(lane + 32 * j, nc - 1));
    }
    if constexpr (STAGED) {   // every column is summed once, for all warps
        float4 *sum_s = S_s + sa.s_rows * nc;
        for (int c = tid; c < nc; c += kSenseThreads) {
            float4 v[kMeanRowBlocks], s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int b = 0; b < kMeanRowBlocks; ++b)
                v[b] = b < sa.blocks ? ld_dep4(sa.x + (size_t)b * d + col0 + 4 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int b = 0; b < kMeanRowBlocks; ++b) { s.x += v[b].x; s.y += v[b].y; s.z += v[b].z; s.w += v[b].w; }
            sum_s[c] = make_float4(s.x * sa.inv_n, s.y * sa.inv_n, s.z * sa.inv_n, s.w * sa.inv_n);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSenseMaxChunks; ++j) xv[j] = lane + 32 * j < nc ? sum_s[lane + 32 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
#pragma unroll
        for (int j = 0; j < kSenseMaxChunks; ++j)
            xv[j] = lane + 32 * j < nc ? ld_dep4(sa.x + (size_t)t * d + col0 + 4 * (lane + 32 * j)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < kSenseMaxChunks; ++j) {
        ss += xv[j].x * xv[j].x + xv[j].y * xv[j].y + xv[j].z * xv[j].z + xv[j].w * xv[j].w;
        if (norm && j < nch) { xv[j].x *= gm[j].x; xv[j].y *= gm[j].y; xv[j].z *= gm[j].z; xv[j].w *= gm[j].w; }
    }
    auto dot = [](const float4 &s, const float4 &v, float a) { return fmaf(s.w, v.w, fmaf(s.z, v.z, fmaf(s.y, v.y, fmaf(s.x, v.x, a)))); };
    // four rows: their reductions interleave; lane q stores row q's
    auto finish = [&](float (&acc)[4], int r0, int end) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = warp_sum(acc[q]);
        if (lane < 4) {
            const int r = r0 + lane * kSenseWarps;
            const float v = lane == 0 ? acc[0] : lane == 1 ? acc[1] : lane == 2 ? acc[2] : acc[3];
            if (r < end) st_remote(remote_smem(&part_s[rank][r], 0), v);
        }
    };
    // (columns past nc repeat the last one with x = 0, rows past the last repeat it and are not stored)
#pragma unroll 1
    for (int r0 = warp; r0 < sa.s_rows; r0 += 4 * kSenseWarps) {
        float acc[4] = {};
        const float4 *row[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) row[q] = S_s + min(r0 + q * kSenseWarps, r0 + (sa.s_rows - 1 - r0) / kSenseWarps * kSenseWarps) * nc;
#pragma unroll
        for (int j = 0; j < kSenseMaxChunks; ++j) {
            if (j >= nch) break;
            const int c = min(lane + 32 * j, nc - 1);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = dot(row[q][c], xv[j], acc[q]);
        }
        finish(acc, r0, sa.s_rows);
    }
    if constexpr (!ALL) {
#pragma unroll 1
        for (int r0 = x0; r0 < m; r0 += 4 * kSenseWarps) {
            float acc[4] = {};
            if (r0 == x0) {
#pragma unroll
                for (int q = 0; q < kSenseExtra; ++q)
#pragma unroll
                    for (int j = 0; j < kSenseMaxChunks; ++j)
                        if (x0 + q * kSenseWarps < m && j < nch) acc[q] = dot(ex[q][j], xv[j], acc[q]);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = r0 + q * kSenseWarps;
                if (r >= m || (r0 == x0 && q < kSenseExtra)) continue;
#pragma unroll
                for (int j = 0; j < kSenseMaxChunks; ++j)
                    if (j < nch) acc[q] = dot(__ldg(reinterpret_cast<const float4 *>(sa.S + (size_t)r * d + col0) + min(lane + 32 * j, nc - 1)), xv[j], acc[q]);
            }
            finish(acc, r0, m);
        }
    }
    if (warp == 0 && norm) {
        ss = warp_sum(ss);
        if (lane < kSenseCtas) st_remote(remote_smem(&ss_s[rank], lane), ss);
    }
    cluster_arrive();
    cluster_wait();
    float rscale = 1.f;
    if (norm) {
        float tot = 0.f;
#pragma unroll
        for (int r = 0; r < kSenseCtas; ++r) tot += ss_s[r];
        rscale = rsqrtf(tot / (float)d + sa.eps);
    }
    if (sa.n_out != nullptr && warp == kSenseWarps - 1) {
#pragma unroll
        for (int j = 0; j < kSenseMaxChunks; ++j)
            if (lane + 32 * j < nc)
                *reinterpret_cast<float4 *>(sa.n_out + (size_t)t * d + col0 + 4 * (lane + 32 * j)) =
                    make_float4(xv[j].x * rscale, xv[j].y * rscale, xv[j].z * rscale, xv[j].w * rscale);
    }
    if (rank != 0 || tid >= GP) return;
    const int g = tid;
    recover_row<NW, KC, 1, PLAIN, true>(
        rs, a, SharedSource{M_s, phi_s, G, pitch},
        [&](auto &sm) {
            for (int i = g; i < m; i += GP) {
                float y = 0.f;
#pragma unroll
                for (int r = 0; r < kSenseCtas; ++r) y += part_s[r][i];
                y *= rscale;
                sm.y[i] = y;
                sa.y_out[(size_t)t * m + i] = y;
            }
        },
        nullptr, g, t, phc);
}

// A plain step whose rows of S do not all fit takes the form for options.  The list goes in steps
// of 8 slots in every form (in steps of 16, 24 of 128 groups of d = 4096, m = 64: 31.3 and 28.8 us a step, with a warm start 27.9 and 25.2).
// One form for options whether the rows fit or not: a step with drift, 12 of 48 groups of d = 2048, four tokens 24.4 us, with two forms and
// recover_init ahead of the wait 23.0; 10 of 40 of d = 1024, one token 15.7 and 15.3; 22 of 86 of d = 5120 29.4 and 28.5.
template <int NW, int KC> SenseFn sense_fn_form(SenseKind kind, bool all) {
    if (kind == kSenseStaged) return sense_recover_kernel<NW, KC, true, true, 0, false>;
    if (kind == kSensePlain && all) return sense_recover_kernel<NW, KC, false, true, 0, true>;
    if (kind == kSensePlainNorm && all) return sense_recover_kernel<NW, KC, false, true, 1, true>;
    return all ? sense_recover_kernel<NW, KC, false, false, 2, true> : sense_recover_kernel<NW, KC, false, false, 2, false>;
}
// k <= G <= 32 NW: the lists a width can meet.  The dense form (65 groups at least) has the prompt's kind only.
template <int NW> SenseFn sense_fn_kc(int k, SenseKind kind, bool all) {
    const int kc = recover_kc(k);
#define CS_SENSE(KC) if (kc == KC) return sense_fn_form<NW, KC>(kind, all)
    CS_SENSE(1); CS_SENSE(2); CS_SENSE(3); CS_SENSE(4);
    if constexpr (NW > 1) { CS_SENSE(5); CS_SENSE(6); CS_SENSE(7); CS_SENSE(8); }
#undef CS_SENSE
    if constexpr (NW > 2) return sense_recover_kernel<NW, 0, true, true, 0, false>;
    return nullptr;
}

}  // namespace cs
