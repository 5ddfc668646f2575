// step_run.cuh -- consecutive local steps with no average between them in one
// pass over the states (mtdao_run).
//
// A single step moves every state through HBM twice for 4 or 2 bytes of new
// gradient.  When a caller hands over the gradients of many steps at once,
// a step depends on nothing but the element's own states and gradients until
// the next average, so the states stay in registers from the first step to
// the last: 8 bytes per state and element once, plus every step's gradients.
//
// A warp holds 128 consecutive elements of one replica, a lane four of them
// in every state; the next step's gradient is on its way while a step is
// computed.
//
// Bound by the update's arithmetic once a launch takes more than a few steps:
// 54 instructions an element and step for Adam with two momenta (profiled,
// M = 4, n = 2^20, 16 steps), most of them in the IEEE square root and
// division.  So what counts is warps to switch between.  Round of 16 steps of
// that size, the last one with its averages a launch of its own: 267 us as
// single steps, 164 at 83 registers a thread, 119 at 64 (4 blocks an SM), 107
// here (5 blocks, one gradient ahead; 117-121 with 4 to 6 blocks and two to
// four gradients ahead).  The averages in the same kernel (a block
// of M warps, the due states meeting in shared memory) took 141 to 166.
// 48 registers spill 44 to 84 bytes for Adam with N = 3 and 4, 16 to 32 for ADOPT,
// which costs less than the fifth block brings on large states (M = 4, us, single
// steps / 5 / 4 blocks: rounds of 16, n = 2^20 Adam N = 3 393 / 114 / 111, N = 4 532
// / 129 / 124, ADOPT N = 3 408 / 124 / 125, N = 4 529 / 136 / 137, SGDM N = 4 364 /
// 71 / 71; of 4, n = 30M Adam N = 3 3025 / 1533 / 1554, ADOPT N = 3 3053 / 1533 /
// 1581).
#pragma once

#include "step_kernels.cuh"

namespace mtdao {

constexpr int kRunChunk = 128;           // elements of one warp

// Four gradient values as they lie in memory, widened when they are used.
template <int GDT>
struct RunGrad;
template <>
struct RunGrad<MTDAO_F32> {
    float4 w;
    __device__ __forceinline__ void load(const char *p) { w = __ldcs(reinterpret_cast<const float4 *>(p)); }
    __device__ __forceinline__ void widen(float (&g)[4]) const { to_array(w, g); }
};
template <>
struct RunGrad<MTDAO_BF16> {
    uint2 w;
    __device__ __forceinline__ void load(const char *p) { w = __ldcs(reinterpret_cast<const uint2 *>(p)); }
    __device__ __forceinline__ void widen(float (&g)[4]) const {
        g[0] = __uint_as_float(w.x << 16);
        g[1] = __uint_as_float(w.x & 0xffff0000u);
        g[2] = __uint_as_float(w.y << 16);
        g[3] = __uint_as_float(w.y & 0xffff0000u);
    }
};

// The steps of one lane's four elements, from the states in memory; the new
// states in s.  e: the lane's first element over all replicas, m: its replica.
template <int BASE, int N, int GDT, bool GUARD>
__device__ __forceinline__ void run_steps(const RunArgs &a, int64_t e, int m,
                                          float (&s)[kNumStates<BASE, N>][4]) {
    constexpr int kStates = kNumStates<BASE, N>;
    constexpr int kGradBytes = GDT == MTDAO_F32 ? 4 : 2;
    const char *g_at = static_cast<const char *>(a.grads) + e * kGradBytes;
    RunGrad<GDT> next;
    next.load(g_at);
#pragma unroll
    for (int st = 0; st < kStates; ++st) to_array(ld_state(a.arena + st * a.stride + e), s[st]);

#pragma unroll 1
    for (int k = 0; k < a.count; ++k) {
        float g[4];
        next.widen(g);
        if (k + 1 < a.count) next.load(g_at + (k + 1) * a.grad_stride);
        StepScalars sc = a.sc;
        sc.neg_lr = a.steps[k].neg_lr;
        sc.sv = a.steps[k].sv;
        sc.clip_c = a.steps[k].clip_c;
#pragma unroll
        for (int j = 0; j < N; ++j) sc.k[j] = a.steps[k].k[j];
        const float scale = a.clip_scale != nullptr ? __ldg(a.clip_scale + k * a.M + m) : 1.0f;
        float gt[4], acc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = step_acc_init<BASE>(sc, g[i], scale);
#pragma unroll
        for (int i = 0; i < kStates; ++i) {
            const int st = state_order<BASE, N>(i);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                update_state<BASE, N, GUARD>(sc, st, g[q], scale, gt[q], acc[q], s[st][q]);
        }
    }
}

template <int BASE, int N, int GDT>
__global__ void __launch_bounds__(kThreads, 5) step_run_kernel(const __grid_constant__ RunArgs a) {
    constexpr int kStates = kNumStates<BASE, N>;
    const int64_t warp = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    int64_t e = warp * kRunChunk;
    if (e >= a.stride) return;
    const int m = static_cast<int>(e / a.n_padded);
    e += 4 * (threadIdx.x & 31);

    // Infinite states are rare and cost an instruction or two per state and
    // step to look for.  Left alone they become NaN (ema_decay), and a NaN
    // stays in its state to the last step: nothing is written before that is
    // looked for, and where one came up the steps are taken again with the
    // guard (which leaves a NaN where there is to be one).
    float s[kStates][4];
    run_steps<BASE, N, GDT, false>(a, e, m, s);
    bool nan = false;
#pragma unroll
    for (int st = 0; st < kStates; ++st)
#pragma unroll
        for (int q = 0; q < 4; ++q) nan = nan || s[st][q] != s[st][q];
    if (nan) run_steps<BASE, N, GDT, true>(a, e, m, s);
#pragma unroll
    for (int st = 0; st < kStates; ++st) st_state(a.arena + st * a.stride + e, from_array(s[st]));
}

template <int BASE, int N, int GDT>
cudaError_t launch_step_run_t(const RunArgs &a, cudaStream_t stream) {
    const int64_t warps = a.stride / kRunChunk;
    const int64_t grid = (warps + kThreads / 32 - 1) / (kThreads / 32);
    if (grid > 0x7fffffff) return cudaErrorInvalidValue;
    step_run_kernel<BASE, N, GDT><<<static_cast<unsigned>(grid), kThreads, 0, stream>>>(a);
    return cudaGetLastError();
}

template <int BASE>
cudaError_t launch_step_run_base(int n_mom, int gdt, const RunArgs &a, cudaStream_t st) {
#define MTDAO_RUN_CASE(NN)                                                          \
    case NN:                                                                        \
        return gdt == MTDAO_F32 ? launch_step_run_t<BASE, NN, MTDAO_F32>(a, st)     \
                                : launch_step_run_t<BASE, NN, MTDAO_BF16>(a, st);
    switch (n_mom) {
        MTDAO_RUN_CASE(1)
        MTDAO_RUN_CASE(2)
        MTDAO_RUN_CASE(3)
        MTDAO_RUN_CASE(4)
        default:
            return cudaErrorInvalidValue;
    }
#undef MTDAO_RUN_CASE
}

}  // namespace mtdao
