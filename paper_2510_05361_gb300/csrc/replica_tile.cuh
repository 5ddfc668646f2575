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

// Replica means of the n_cols columns of a block's tiles into mean[p], column
// p = k * S + c being column c of the k-th tile: tile_of(k) is where that tile
// [M][S] begins; the bits of replica_mean.cuh (with its plain mean where the
// compensated one is NaN).
//
// V > 0: a lane takes V neighbouring columns and runs both compensated parts
// over the replicas in order (1 .. h-1 and h .. M-1, h = M / 2), one replica of
// each part a step, so that the two chains overlap.  Against a pair of lanes
// per four columns (a part each, joined by shuffles; most of the fused step's
// time above HBM's was its instructions: 52 of 177 an element at M = 8), fused
// step, us, pair -> here with V = 1 (V = 4): M = 8, n = 20M, ADOPT N = 2, bf16
// 832 -> 785 (793), Adam N = 3 1051 -> 1014 (1010); M = 9, n = 2^23 511 -> 483
// (483); M = 16, ADOPT 686 -> 659 (671); M = 12 529 -> 511 (496); M = 64, n = 1M
// 346 -> 326 (439).  (Half of it is the item loops of step_sync_wide.cuh.)
// V = 0: a pair of half-warps takes a column a lane, one part each, joined by a
// shuffle: twice the lanes on chains that are long and tiles that are narrow
// (average, M = 256, n = 400k 370 -> 367 us, n = 1000 8.0 -> 6.2, M = 1024, n =
// 100k 452 -> 378; fused, M = 100 359 -> 353).  kSplitMeansM: M from which it is
// always taken.
constexpr int kSplitMeansM = 65;

//
// POW2: M is a power of two, and the division by it is the product with its
// reciprocal: the same bits, but a division of zero (replicas that are equal)
// leaves the fast path of the divide (fused step, M = 4, n = 20M, Adam N = 3, every
// state equal 607 us -> 512, apart 516 -> 510; SGDM N = 2, n = 30M 555 -> 484).
// Not with V = 0, whose small blocks feel a second copy of the loops (M = 16 to 64,
// n = 250 to 8000 2 % slower in the mean, up to 15 %).
template <int V, bool POW2, typename TileOf>
__device__ __forceinline__ void tile_means_of(TileOf tile_of, int M, int log2_s, int n_cols, float *mean) {
    const int S = 1 << log2_s;
    const int h = M / 2;
    const float fM = static_cast<float>(M);
    auto from_parts = [inv = 1.0f / fM, fM](float s0, float part_a, float part_b) {
        if constexpr (POW2) {
            const float q = (part_a + part_b) * inv;
            return q == 0.0f ? s0 : s0 + q;
        } else {
            return replica_mean_from_parts(s0, part_a, part_b, fM);
        }
    };
    auto column = [&](int p) { return tile_of(p >> log2_s) + (p & (S - 1)); };
    if constexpr (V == 0) {
        const int part = (threadIdx.x >> 4) & 1;
        const int lo = part ? (h > 1 ? h : 1) : 1, hi = part ? M : h;
        // every lane of a warp with a column left goes round (the shuffle)
        for (int p0 = static_cast<int>(threadIdx.x >> 5) * 16; p0 < n_cols; p0 += static_cast<int>(blockDim.x >> 1)) {
            const int p = p0 + static_cast<int>(threadIdx.x & 15);
            const float *base = column(p < n_cols ? p : n_cols - 1);
            const float s0 = *base;
            DiffSum sum(s0);
#pragma unroll 4
            for (int m = lo; m < hi; ++m) sum.add(base[m * S]);
            const float mine = sum.partial();
            const float other = __shfl_xor_sync(0xffffffffu, mine, 16);
            if (p < n_cols && part == 0) {
                float v = from_parts(s0, mine, other);
                if (v != v) {                    // non-finite values: the plain mean
                    float plain = s0;
                    for (int m = 1; m < M; ++m) plain += base[m * S];
                    v = plain / fM;
                }
                mean[p] = v;
            }
        }
    } else {
        for (int p = V * static_cast<int>(threadIdx.x); p < n_cols; p += V * static_cast<int>(blockDim.x)) {
            const float *base = column(p);
            float s0[V], v[V], w[V];
            ld_shared_v<V>(base, s0);
            DiffSum pa[V], pb[V];
#pragma unroll
            for (int k = 0; k < V; ++k) pa[k] = pb[k] = DiffSum(s0[k]);
            const float *at = base + S;              // replica 1 + j of part A, h + j of part B
            const int to_b = (h - 1) * S;
#pragma unroll 2
            for (int j = 1; j < h; ++j, at += S) {
                ld_shared_v<V>(at, v);
                ld_shared_v<V>(at + to_b, w);
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    pa[k].add(v[k]);
                    pb[k].add(w[k]);
                }
            }
            for (int m = h > 1 ? 2 * h - 1 : 1; m < M; ++m) {        // part B's last one or two
                ld_shared_v<V>(base + m * S, v);
#pragma unroll
                for (int k = 0; k < V; ++k) pb[k].add(v[k]);
            }
            bool nan = false;
#pragma unroll
            for (int k = 0; k < V; ++k) {
                v[k] = from_parts(s0[k], pa[k].partial(), pb[k].partial());
                nan = nan || v[k] != v[k];
            }
            if (nan) {                               // non-finite values: the plain mean (replica_mean.cuh)
#pragma unroll
                for (int k = 0; k < V; ++k) {
                    float plain = s0[k];
                    for (int m = 1; m < M; ++m) plain += base[m * S + k];
                    v[k] = mean_or_plain(v[k], plain, fM);
                }
            }
#pragma unroll
            for (int k = 0; k < V; ++k) mean[p + k] = v[k];
        }
    }
}

template <int V, typename TileOf>
__device__ __forceinline__ void tile_means(TileOf tile_of, int M, int log2_s, int n_cols, float *mean) {
    if (V != 0 && (M & (M - 1)) == 0)
        tile_means_of<V, V != 0>(tile_of, M, log2_s, n_cols, mean);
    else
        tile_means_of<V, false>(tile_of, M, log2_s, n_cols, mean);
}

// The means of one tile.
template <int V>
__device__ __forceinline__ void tile_means(const float *tile, int M, int log2_s, float *mean) {
    tile_means<V>([=](int) { return tile; }, M, log2_s, 1 << log2_s, mean);
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

// Opts a kernel in to more than the default 48 KB of dynamic shared memory: to
// the most that any tile takes, whatever this launch needs.  The limit belongs
// to the kernel, not to the launch, so a limit of this launch's size would
// refuse a larger tile that another thread is about to launch.
template <typename Kernel>
inline cudaError_t allow_shared(Kernel kernel, size_t smem) {
    if (smem <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(kSharedPerSm - kSharedReserved));
}

}  // namespace mtdao
