// stats_wide.cu -- the cross-worker diagnostics of section 4.1 for more
// replicas than a thread holds (9 <= M <= 1024; large states of 450 replicas and
// more are streamed, reduce_kernels.cu).
//
// A block takes a run of consecutive tiles, S columns of all M replicas each:
// copies a tile to shared memory (cp.async), forms its replica means
// (tile_means: the bits of the standalone average) and adds every replica's
// sums against the mean; the sync diagnostics then store the mean over the
// replicas (the average itself).  Every replica value is read from HBM once.
// What overlaps the copies of a block is the work of the others on its SM.
//
// Sums are bit-reproducible: a position's four elements are summed in fp32,
// each thread accumulates its positions with Kahan compensation, the L lanes of a
// replica combine theirs by a fixed shuffle pattern (kahan.cuh), the block writes
// one row in fp64, and launch_stats_finalize adds the rows in a fixed order.
#include <cuda_runtime.h>
#include <cstdint>

#include "kahan.cuh"
#include "mtdao_internal.h"
#include "replica_tile.cuh"
#include "step_kernels.cuh"

namespace mtdao {

namespace {

constexpr int kStatsTileThreads = 256;

struct StatsTileArgs {
    float *arena;                    // state sel[blockIdx.y] at arena + sel * stride, [M][n]
    const float *anchor;             // change diagnostics: [n]
    float *new_anchor[2 + MTDAO_MAX_MOM];    // sync diagnostics: [n] copy of the mean, or nullptr
    double *partial;                 // [state][Q][gridDim.x]
    int64_t n, stride;
    int32_t sel[2 + MTDAO_MAX_MOM];
    int32_t M;
    int32_t tiles;                   // tiles of a run
    int32_t log2_s, log2_l;          // columns of a tile, lanes of a replica
};

// CHANGE = false, sync diagnostics (Q = 2 + 2M):
//   q = 0          sum_m sum_i (s_m - s_bar)^2
//   q = 1          sum_i s_bar^2
//   q = 2 + m      sum_i s_m^2
//   q = 2 + M + m  sum_i s_m * s_bar
// CHANGE = true, change of x against the anchor a, read-only (Q = 2M + 2):
//   q = m          sum_i (x_m - a)^2
//   q = M + m      sum_i (x_m - a) * (x_bar - a)
//   q = 2M         sum_i (x_bar - a)^2
//   q = 2M + 1     sum_i a^2
// Thread t takes the rows (replicas) t / L + k * blockDim / L, k < R.
template <bool CHANGE, int R, int V>
__global__ void __launch_bounds__(kStatsTileThreads) stats_tile_kernel(const __grid_constant__ StatsTileArgs a) {
    extern __shared__ __align__(16) float smem[];
    const int M = a.M;
    const int S = 1 << a.log2_s;
    const int log2_p = a.log2_s - 2;
    const int L = 1 << a.log2_l;
    const int items = M << log2_p;
    const int t = threadIdx.x;
    const int lane = t & (L - 1);
    const int row0 = t >> a.log2_l;
    const int row_step = static_cast<int>(blockDim.x) >> a.log2_l;
    const int64_t n = a.n;
    float *base = a.arena + static_cast<int64_t>(a.sel[blockIdx.y]) * a.stride;
    float *tile = smem;                          // [M][S]
    float *mean = smem + M * S;                  // [S]
    float *anc = mean + S;                       // [S] (CHANGE)
    Kahan own[R], cross[R];                      // s_m^2 and s_m s_bar, or (x_m - a)^2 and (x_m - a)(x_bar - a)
    Kahan all, ref;                              // (s_m - s_bar)^2 and s_bar^2, or (x_bar - a)^2 and a^2

    const int64_t n_tiles = n >> a.log2_s;
    const int64_t first = static_cast<int64_t>(blockIdx.x) * a.tiles;
    const int64_t last = first + a.tiles < n_tiles ? first + a.tiles : n_tiles;
    for (int64_t k = first; k < last; ++k) {
        const int64_t col0 = k << a.log2_s;
        for (int i = t; i < items; i += static_cast<int>(blockDim.x))
            cp_async16(tile + 4 * i, base + (i >> log2_p) * n + col0 + 4 * (i & ((1 << log2_p) - 1)));
        if (CHANGE && t < (1 << log2_p)) cp_async16(anc + 4 * t, a.anchor + col0 + 4 * t);
        cp_async_commit();
        cp_async_wait<0>();                      // this thread's copies have landed
        __syncthreads();                         // ... and every thread's
        tile_means<V>(tile, M, a.log2_s, mean);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < R; ++j) {
            const int r = row0 + j * row_step;
            if (r >= M) break;
            for (int c = 4 * lane; c < S; c += 4 * L) {
                float p0 = 0.0f, p1 = 0.0f, p2 = 0.0f, p3 = 0.0f;     // this position's four elements
                float x[4], mb[4];
                to_array(*reinterpret_cast<const float4 *>(tile + r * S + c), x);
                to_array(*reinterpret_cast<const float4 *>(mean + c), mb);
                if constexpr (CHANGE) {
                    float av[4];
                    to_array(*reinterpret_cast<const float4 *>(anc + c), av);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float loc = x[q] - av[q], glob = mb[q] - av[q];
                        p0 = fmaf(loc, loc, p0);
                        p1 = fmaf(loc, glob, p1);
                        p2 = fmaf(glob, glob, p2);
                        p3 = fmaf(av[q], av[q], p3);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float dv = x[q] - mb[q];
                        p0 = fmaf(x[q], x[q], p0);
                        p1 = fmaf(x[q], mb[q], p1);
                        p2 = fmaf(dv, dv, p2);
                        p3 = fmaf(mb[q], mb[q], p3);
                    }
                }
                own[j].add(p0);
                cross[j].add(p1);
                if (!CHANGE || r == 0) all.add(p2);
                if (r == 0) ref.add(p3);
            }
        }
        if constexpr (!CHANGE) {
            for (int i = t; i < items; i += static_cast<int>(blockDim.x)) {
                const int f = i & ((1 << log2_p) - 1);
                st_state(base + (i >> log2_p) * n + col0 + 4 * f, *reinterpret_cast<const float4 *>(mean + 4 * f));
            }
            float *to = a.new_anchor[blockIdx.y];
            if (to != nullptr && t < (1 << log2_p))
                st_state(to + col0 + 4 * t, *reinterpret_cast<const float4 *>(mean + 4 * t));
        }
        __syncthreads();                         // the tile and the means are rewritten next
    }

    const int Q = 2 + 2 * M;
    double *out = a.partial + static_cast<int64_t>(blockIdx.y) * Q * gridDim.x + blockIdx.x;
    auto put = [&](int q, double v) { out[static_cast<int64_t>(q) * gridDim.x] = v; };
    const int own_at = CHANGE ? 0 : 2;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int r = row0 + j * row_step;
        const double v = lanes_sum2_wide(own[j], cross[j], L);
        if (r < M && lane < 2) put(own_at + lane * M + r, v);
    }
    if constexpr (CHANGE) {                      // both in the lanes of replica 0
        if (t < 32) {
            const double v = lanes_sum2_wide(all, ref, L);
            if (t < 2) put(2 * M + t, v);
        }
    } else {
        __shared__ double part[kStatsTileThreads / 32];
        // s_bar^2 lies in the lanes of replica 0, in the first warp
        const double v = lanes_sum2_wide(all, ref, 32);
        if ((t & 31) == 0) part[t >> 5] = v;
        __syncthreads();
        if (t == 0) {
            double total = 0.0;
            for (int i = 0; i < static_cast<int>(blockDim.x >> 5); ++i) total += part[i];
            put(0, total);
        }
        if (t == 1) put(1, v);
    }
}

struct StatsTileShape {
    int log2_s, log2_l, R, threads, tiles;
    int64_t runs;                    // blocks of one state
    size_t smem;
};

// Columns, lanes of a replica, threads and tiles of a run (diagnostics of a
// round's end -- change of x, then the average of every state with its sums --
// in us; the previous kernels, one-pass in rows of 128 to 256 bytes with
// persistent blocks up to M = 64 and two passes above, first).
//   Columns: 256 up to M = 12 (M = 9, Adam N = 1, n = 8M: 534 -> 427), 128 up
//   to 16 (M = 16, Adam N = 2, n = 8M: 942 -> 758), 64 up to 256 (M = 32, n =
//   4M: 781 -> 612; M = 64, n = 2M: 709 -> 617; M = 128, n = 600k: 1102 -> 497; M
//   = 256, n = 400k: 1073 -> 635), 32 above, where 64 leave an SM two or three
//   small blocks (change, M = 320, n = 1.25M 911 -> 553, M = 257, n = 3.1M 1339
//   -> 1022; average with sums, M = 384, n = 521k, 3 states 1457 -> 1044) but
//   for small states (change, M = 257, n = 29k 64 columns 19, 32 24); fewer
//   where two tiles would not fit an SM or the SMs would not have one each.
//   Lanes and threads: the fewer, the more rows a thread takes and the less
//   there is to combine at a run's end (M = 64, means by lane pairs: 2 lanes and
//   128 threads 639, 8 lanes 683, 512 threads 1120).
//   Tiles: runs enough for 8 blocks an SM, 8 at most, so that the tiles under
//   way lie close together (M = 64: 640, runs of 32 675; M = 100, n = 75k, runs
//   of 1 to 2: 231 -> 56, of 32 254); as many columns (512) where the tiles are
//   narrower (M = 1024, n = 100k: 1305 -> 998 in runs of 6, 1033 of 12).
//   Workspace: 16 bytes a run and replica, under 1 % of the states in runs of 512
//   columns, more on small states (6 % at M = 100, n = 75k with runs of one tile of
//   64 columns, half of them with tiles of 8).
StatsTileShape stats_tile_shape(int num_sms, int64_t n, int n_sel, int M) {
    StatsTileShape w;
    auto bytes = [&](int log2_s) { return static_cast<size_t>(M + 2) * sizeof(float) << log2_s; };
    w.log2_s = M <= 12 ? 8 : (M <= 16 ? 7 : (M <= 256 || (n >> 6) * n_sel < 4 * num_sms ? 6 : 5));
    while (w.log2_s > 3 &&
           (2 * (bytes(w.log2_s) + kSharedReserved) > kSharedPerSm || (n >> w.log2_s) * n_sel < num_sms))
        --w.log2_s;
    w.smem = bytes(w.log2_s);
    w.log2_l = M <= 16 ? 2 : 1;                  // 2^log2_l <= S / 4 for every S
    if (w.log2_l > w.log2_s - 2) w.log2_l = w.log2_s - 2;
    w.R = 1;
    while (w.R < 8 && (M << w.log2_l) > w.R * 128) w.R *= 2;
    w.threads = (((M << w.log2_l) + w.R - 1) / w.R + 31) / 32 * 32;
    const int64_t n_tiles = n >> w.log2_s;
    const int64_t per = n_tiles * n_sel / (8 * static_cast<int64_t>(num_sms));
    const int64_t most = w.log2_s >= 6 ? 8 : 512 >> w.log2_s;
    w.tiles = static_cast<int>(per < 1 ? 1 : (per > most ? most : per));
    w.runs = (n_tiles + w.tiles - 1) / w.tiles;
    return w;
}

template <bool CHANGE, int R, int V>
cudaError_t launch_stats_tile_t(const StatsTileArgs &a, const StatsTileShape &w, int n_sel, cudaStream_t stream) {
    auto kernel = stats_tile_kernel<CHANGE, R, V>;
    if (const cudaError_t e = allow_shared(kernel, w.smem); e != cudaSuccess) return e;
    kernel<<<dim3(static_cast<unsigned>(w.runs), n_sel), w.threads, w.smem, stream>>>(a);
    return cudaGetLastError();
}

template <bool CHANGE>
cudaError_t launch_stats_tile(StatsTileArgs &a, int n_sel, int num_sms, size_t partial_cap, double *stats,
                              cudaStream_t stream) {
    const int Q = 2 + 2 * a.M;
    const StatsTileShape w = stats_tile_shape(num_sms, a.n, n_sel, a.M);
    if (w.runs > 0x7fffffff || static_cast<size_t>(w.runs) * n_sel * Q > partial_cap) return cudaErrorInvalidValue;
    a.log2_s = w.log2_s;
    a.log2_l = w.log2_l;
    a.tiles = w.tiles;
    cudaError_t e;
    // R = 1 is M <= 64 (tile_means, with the rows' sums compensated once a tile:
    // M = 9 380 us with two columns a lane, 402 with one, 392 with four; M = 64
    // 616 with one, 651 with two)
    switch (w.R) {
        case 1:
            e = a.M <= 16 ? launch_stats_tile_t<CHANGE, 1, 2>(a, w, n_sel, stream)
                          : launch_stats_tile_t<CHANGE, 1, 1>(a, w, n_sel, stream);
            break;
        case 2: e = launch_stats_tile_t<CHANGE, 2, 0>(a, w, n_sel, stream); break;
        case 4: e = launch_stats_tile_t<CHANGE, 4, 0>(a, w, n_sel, stream); break;
        default: e = launch_stats_tile_t<CHANGE, 8, 0>(a, w, n_sel, stream); break;
    }
    if (e != cudaSuccess) return e;
    return launch_stats_finalize(a.partial, w.runs, Q, n_sel, CHANGE ? 0 : a.M, stats, stream);
}

}  // namespace

size_t tile_stats_partial_capacity(int num_sms, int64_t n_padded, int n_states, int M) {
    int64_t most = 0;
    for (int k = 1; k <= n_states; ++k) {
        const int64_t rows = stats_tile_shape(num_sms, n_padded, k, M).runs * k;
        if (rows > most) most = rows;
    }
    return static_cast<size_t>(most) * (2 + 2 * static_cast<size_t>(M));
}

cudaError_t launch_sync_stats_tile(const SyncArgs &s, int num_sms, double *partial, size_t partial_cap,
                                   double *stats, cudaStream_t stream) {
    if (s.n_sel <= 0) return cudaSuccess;
    StatsTileArgs a = {};
    a.arena = s.arena;
    a.partial = partial;
    a.n = s.n_padded;
    a.stride = s.stride;
    a.M = s.M;
    for (int k = 0; k < s.n_sel; ++k) {
        a.sel[k] = s.sel[k];
        a.new_anchor[k] = s.anchor[k];
    }
    return launch_stats_tile<false>(a, s.n_sel, num_sms, partial_cap, stats, stream);
}

cudaError_t launch_pseudo_grad_stats_tile(const float *x, const float *anchor, int64_t n, int M, int num_sms,
                                          double *partial, size_t partial_cap, double *stats,
                                          cudaStream_t stream) {
    StatsTileArgs a = {};
    a.arena = const_cast<float *>(x);            // not written
    a.anchor = anchor;
    a.partial = partial;
    a.n = n;
    a.M = M;
    return launch_stats_tile<true>(a, 1, num_sms, partial_cap, stats, stream);
}

}  // namespace mtdao
