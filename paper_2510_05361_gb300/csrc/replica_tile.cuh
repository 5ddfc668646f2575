// replica_tile.cuh -- tiles of all M replicas in shared memory: S consecutive
// columns of every replica, and their replica means.  Shared by the fused
// step (step_sync_wide.cuh), the standalone average (reduce_kernels.cu) and
// the diagnostics (stats_wide.cu).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

#include "replica_mean.cuh"
#include "step_kernels.cuh"

namespace mtdao {

constexpr size_t kSharedPerSm = 227 * 1024;      // shared memory of an SM
constexpr size_t kSharedReserved = 1024;         // ... of it reserved for each resident block

// V consecutive floats of shared memory.
template <int V>
__device__ __forceinline__ void ld_shared_v(const float *p, float (&v)[V]) {
    if constexpr (V == 4) {
        to_array(*reinterpret_cast<const float4 *>(p), v);
    } else if constexpr (V == 2) {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x;
        v[1] = t.y;
    } else {
        v[0] = *p;
    }
}

// Replica means of the n_cols columns of a block's tiles into mean[p]
// (column p: tile + (p / S) * M * S + p % S, the replicas at stride
// S = 2^log2_s).  Columns go in groups of V; lanes i and i + 16 of a warp
// take one group and form its two compensated parts of replica_mean.cuh,
// replicas 1 .. h-1 and h .. M-1 in order (h = M / 2), and join them with a
// shuffle: the bits of replica_mean_rt (with its plain mean where the
// compensated one is NaN).  A half-warp reads one row, so no two of its
// lanes meet in a bank.  Every thread of the block calls it (the shuffles
// take whole warps: blockDim.x is a multiple of 32).
template <int V>
__device__ __forceinline__ void tile_means(const float *tile, int M, int log2_s, int n_cols, float *mean) {
    const int h = M / 2;
    const int S = 1 << log2_s;
    const int part = (threadIdx.x >> 4) & 1;
    const int first = V * ((threadIdx.x >> 5) * 16 + (threadIdx.x & 15));
    const int lo = part ? (h > 1 ? h : 1) : 1, hi = part ? M : h;
    for (int p0 = 0; p0 < n_cols; p0 += V * static_cast<int>(blockDim.x >> 1)) {
        if (p0 + V * 16 * static_cast<int>(threadIdx.x >> 5) >= n_cols) break;      // the whole warp is past the end
        const int p = p0 + first;
        const float *base = tile + (p >> log2_s) * M * S + (p & (S - 1));
        float s0[V], mine[V], other[V];
#pragma unroll
        for (int k = 0; k < V; ++k) s0[k] = mine[k] = 0.0f;
        if (p < n_cols) {
            ld_shared_v<V>(base, s0);
            float sum[V], comp[V];
#pragma unroll
            for (int k = 0; k < V; ++k) sum[k] = comp[k] = 0.0f;
#pragma unroll 4
            for (int m = lo; m < hi; ++m) {
                float v[V];
                ld_shared_v<V>(base + m * S, v);
#pragma unroll
                for (int k = 0; k < V; ++k) {            // DiffSum::add
                    const float y = (v[k] - s0[k]) - comp[k];
                    const float t = sum[k] + y;
                    comp[k] = (t - sum[k]) - y;
                    sum[k] = t;
                }
            }
#pragma unroll
            for (int k = 0; k < V; ++k) mine[k] = sum[k] - comp[k];
        }
#pragma unroll
        for (int k = 0; k < V; ++k) other[k] = __shfl_xor_sync(0xffffffffu, mine[k], 16);
        if (p < n_cols && part == 0) {
#pragma unroll
            for (int k = 0; k < V; ++k) {
                float v = replica_mean_from_parts(s0[k], mine[k], other[k], static_cast<float>(M));
                if (v != v) {                    // non-finite values: the plain mean (replica_mean.cuh)
                    float plain = s0[k];
                    for (int m = 1; m < M; ++m) plain += base[m * S + k];
                    v = plain / static_cast<float>(M);
                }
                mean[p + k] = v;
            }
        }
    }
}

// 16- and 8-byte asynchronous global -> shared copies (cp.async) and their
// groups.
__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src) {
    const unsigned dst = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async8(void *smem_dst, const void *gmem_src) {
    const unsigned dst = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Blocks of an SM with this much shared memory each (at least one).
inline int64_t tile_blocks_fit(size_t smem) {
    const int64_t fit = static_cast<int64_t>(kSharedPerSm / (smem + kSharedReserved));
    return fit < 1 ? 1 : fit;
}

// Opts a kernel in to more than the default 48 KB of dynamic shared memory.
template <typename Kernel>
inline cudaError_t allow_shared(Kernel kernel, size_t smem) {
    if (smem <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
}

}  // namespace mtdao
