// The sensing launch as the host sees it; the kernel is sense_kernel.cuh.
#pragma once
#include "recover_core.cuh"

namespace cs {

constexpr int kSenseCtas = 8;
constexpr int kSenseThreads = 256;
constexpr int kSenseWarps = kSenseThreads / 32;
constexpr int kSenseMaxChunks = kMaxD / kSenseCtas / 4 / 32;   // float4 columns per lane
constexpr int kSenseSmem = 220 * 1024;                         // dynamic, at most
constexpr int kSenseExtra = 1;                                 // rows of S a warp keeps in registers

struct SenseArgs {
    const float *S, *x, *gamma;
    float eps;
    int d, s_rows;        // s_rows: rows of S that fit in shared memory (the others are read after the wait)
    float *y_out, *n_out;
    int blocks;           // STAGED: x is [blocks, d], and what is sensed is the sum of its rows times inv_n
    float inv_n;
};

typedef void (*SenseFn)(SenseArgs, RecoverArgs);

inline int recover_kc(int k) { return k <= 64 ? (k + 7) / 8 : 0; }
enum SenseKind { kSensePlain, kSensePlainNorm, kSenseOptions, kSenseStaged };
// The kernel for G in (32 (NW - 1), 32 NW].  all: every row of S has its place in shared memory.  A unit of its own per width
// (sense_w1.cu ...): a plan loads the kernels of its own only.
template <int NW> SenseFn sense_fn_kc(int k, SenseKind kind, bool all);

}  // namespace cs
