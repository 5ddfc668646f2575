// reduce_kernels.cu -- replica averaging (outer synchronisation) and the
// per-replica gradient norm used by clip(g, rho).
//
// Averaging (Algorithms 1-3, E_m[.] with averaging as OuterOpt): for every
// selected state and element, the M replica values are read once and the
// mean (replica_mean.cuh) is written back to all M replicas.  Algorithmic traffic: 8 * M bytes
// per element per state.  HBM-bound; one grid row (blockIdx.y) per selected
// state.
//
// Norm: sum_i g[m][i]^2 per replica with a fixed grid and fixed reduction
// order, so the result is bit-reproducible.  Each thread accumulates its
// strided share in fp32 with Kahan compensation, warps and blocks combine in
// fp64, and a second small kernel adds the per-block partials in order.
#include <cuda_runtime.h>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "mtdao_internal.h"
#include "kahan.cuh"
#include "replica_mean.cuh"
#include "replica_tile.cuh"
#include "step_kernels.cuh"

namespace mtdao {

namespace {

// One float4 position of one state per thread, the replicas in registers.
template <int M>
__global__ void __launch_bounds__(kThreads) sync_kernel(const __grid_constant__ SyncArgs a) {
    float *base = a.arena + static_cast<int64_t>(a.sel[blockIdx.y]) * a.stride;
    const int64_t n = a.n_padded;
    const int64_t nv = n / 4;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nv;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t e = 4 * i;
        float r[M][4], mean[4];
#pragma unroll
        for (int m = 0; m < M; ++m) to_array(ld_state(base + m * n + e), r[m]);
#pragma unroll
        for (int k = 0; k < 4; ++k) mean[k] = replica_mean<M>([&](int m) { return r[m][k]; });
        const float4 mv = from_array(mean);
#pragma unroll
        for (int m = 0; m < M; ++m) st_state(base + m * n + e, mv);
        if (a.anchor[blockIdx.y] != nullptr) st_state(a.anchor[blockIdx.y] + e, mv);
    }
}

template <int M>
cudaError_t launch_sync_t(const SyncArgs &a, cudaStream_t stream) {
    // M = 2 .. 14: one float4 position per thread, like the local step's
    // stream_grid (flat 2^27, all states, GB/s against a persistent grid:
    // M = 2 6342 -> 7098, M = 4 6447 -> 7025, M = 8 6546 -> 6941).  At 15 and
    // 16 the replicas take 151-176 registers.
    const int64_t need = (a.n_padded / 4 + kThreads - 1) / kThreads;
    const int64_t gx = need > 0x7fffffff ? 0x7fffffff : need;
    dim3 grid(static_cast<unsigned>(gx), static_cast<unsigned>(a.n_sel));
    sync_kernel<M><<<grid, kThreads, 0, stream>>>(a);
    return cudaGetLastError();
}

constexpr int kSyncTileThreads = 128;

// The average on one tile of S = 4 * 2^log2_p columns of all replicas per
// block: copied to shared memory, the means formed there, stored to every
// replica; the blocks start in index order.  Takes M > 14 (but for what
// stream_replicas names), where a thread that streams the replicas of its
// position (four loads in flight, persistent grid) has one long chain of loads
// behind its sums.  That one -> this, us:
// M = 16, n = 8M, one state 179 -> 152, n = 20k 8.2 -> 4.1; M = 32, n = 5M, 3
// states 620 -> 552 (6.96 TB/s), n = 200k 14.4 -> 8.2; M = 64, n = 2M 504 ->
// 448; M = 256, n = 400k 423 -> 366, n = 1000 65.5 -> 6.2; M = 1024, n = 20k 258
// -> 45.  Bound by HBM; from M = 450 on by the rows of 128 and 64 bytes of the
// tiles that two of them fit on an SM with.
template <int V>
__global__ void __launch_bounds__(kSyncTileThreads) sync_tile_kernel(const __grid_constant__ SyncArgs a, int log2_p) {
    extern __shared__ __align__(16) float smem[];
    const int M = a.M;
    const int S = 4 << log2_p;
    const int items = M << log2_p;
    const int64_t n = a.n_padded;
    float *base = a.arena + static_cast<int64_t>(a.sel[blockIdx.y]) * a.stride + static_cast<int64_t>(blockIdx.x) * S;
    float *mean = smem + M * S;
    for (int i = threadIdx.x; i < items; i += static_cast<int>(blockDim.x))
        cp_async16(smem + 4 * i, base + (i >> log2_p) * n + 4 * (i & ((1 << log2_p) - 1)));
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    tile_means<V>(smem, M, log2_p + 2, mean);
    __syncthreads();
    for (int i = threadIdx.x; i < items; i += static_cast<int>(blockDim.x)) {
        const int f = i & ((1 << log2_p) - 1);
        st_state(base + (i >> log2_p) * n + 4 * f, *reinterpret_cast<const float4 *>(mean + 4 * f));
    }
    float *anchor = a.anchor[blockIdx.y];
    if (anchor != nullptr && threadIdx.x < (1 << log2_p))
        st_state(anchor + static_cast<int64_t>(blockIdx.x) * S + 4 * threadIdx.x,
                 *reinterpret_cast<const float4 *>(mean + 4 * threadIdx.x));
}

size_t sync_tile_bytes(int M, int log2_p) { return (static_cast<size_t>(M + 1) * 4 * sizeof(float)) << log2_p; }

// Columns of a tile (4 * 2^log2_p) of large states: 128 up to M = 32 (M = 16:
// 152 us, 64 columns 195), 64 above (M = 64: 448, 128 columns 451), fewer where
// two tiles would not fit an SM (32 from M = 450, 16 from M = 900).
int sync_tile_log2_p(int M) {
    int log2_p = M <= 32 ? 5 : 4;
    while (log2_p > 1 && 2 * (sync_tile_bytes(M, log2_p) + kSharedReserved) > kSharedPerSm) --log2_p;
    return log2_p;
}

cudaError_t launch_sync_tile(const SyncArgs &a, int num_sms, cudaStream_t stream) {
    // Fewer columns where the SMs would not have a tile each.  128 threads: M =
    // 32 552 us, 256 560-580, 512 824-863.
    int log2_p = sync_tile_log2_p(a.M);
    while (log2_p > 1 && (a.n_padded >> (log2_p + 2)) * a.n_sel < num_sms) --log2_p;
    const size_t smem = sync_tile_bytes(a.M, log2_p);
    auto kernel = a.M < kSplitMeansM ? sync_tile_kernel<1> : sync_tile_kernel<0>;
    if (const cudaError_t e = allow_shared(kernel, smem); e != cudaSuccess) return e;
    const int64_t gx = a.n_padded >> (log2_p + 2);
    if (gx > 0x7fffffff) return cudaErrorInvalidValue;
    kernel<<<dim3(static_cast<unsigned>(gx), static_cast<unsigned>(a.n_sel)), kSyncTileThreads, smem, stream>>>(
        a, log2_p);
    return cudaGetLastError();
}

// Mean of the M replicas at float4 position e of state s: replica_mean.cuh's
// operations in its order, four replicas' loads in flight.
__device__ __forceinline__ float4 replica_mean4(const float *s, int64_t n, int M, int64_t e) {
    float s0[4];
    to_array(ld_state(s + e), s0);
    DiffSum pa[4] = {DiffSum(s0[0]), DiffSum(s0[1]), DiffSum(s0[2]), DiffSum(s0[3])};
    DiffSum pb[4] = {DiffSum(s0[0]), DiffSum(s0[1]), DiffSum(s0[2]), DiffSum(s0[3])};
    float plain[4] = {s0[0], s0[1], s0[2], s0[3]};
    const int h = M / 2;
    for (int m = 1; m < M; m += 4) {
        float r[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (m + u < M) to_array(ld_state(s + (m + u) * n + e), r[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (m + u >= M) break;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (m + u < h) pa[k].add(r[u][k]);
                else pb[k].add(r[u][k]);
                plain[k] += r[u][k];
            }
        }
    }
    float mean[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        mean[k] = mean_or_plain(
            replica_mean_from_parts(s0[k], pa[k].partial(), pb[k].partial(), static_cast<float>(M)), plain[k],
            static_cast<float>(M));
    return from_array(mean);
}

// The average of many replicas of large states (stream_replicas): a thread
// streams the replicas of its float4 position, on a persistent grid.
__global__ void __launch_bounds__(kThreads) sync_stream_kernel(const __grid_constant__ SyncArgs a) {
    float *base = a.arena + static_cast<int64_t>(a.sel[blockIdx.y]) * a.stride;
    const int64_t n = a.n_padded;
    const int64_t nv = n / 4;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nv;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t e = 4 * i;
        const float4 mv = replica_mean4(base, n, a.M, e);
        for (int m = 0; m < a.M; ++m) st_state(base + m * n + e, mv);
        if (a.anchor[blockIdx.y] != nullptr) st_state(a.anchor[blockIdx.y] + e, mv);
    }
}

cudaError_t launch_sync_stream(const SyncArgs &a, int num_sms, cudaStream_t stream) {
    static const int per_sm = blocks_per_sm(sync_stream_kernel);
    const int64_t need = (a.n_padded / 4 + kThreads - 1) / kThreads;
    int64_t gx = static_cast<int64_t>(per_sm) * num_sms / a.n_sel;
    if (gx > need) gx = need;
    if (gx < 1) gx = 1;
    sync_stream_kernel<<<dim3(static_cast<unsigned>(gx), static_cast<unsigned>(a.n_sel)), kThreads, 0, stream>>>(a);
    return cudaGetLastError();
}

// Whether n_sel states of n elements are averaged by threads that stream the
// replicas (rows of 512 bytes a warp, but a chain of loads as long as M) instead
// of by tiles of all of them.  Where tiles have 64 columns or more, never; below,
// once there are columns enough for every thread of the streaming grid.  us,
// tiles / streamed, three states, by columns (n * 3):
//   16 columns: M = 1024 60k 116 / 269, 176k 329 / 378, 351k 652 / 510, 586k
//   1139 / 737, 1.2M 2556 / 1520 (one state 117k 227 / 273, 195k 388 / 379).
//   32 columns, two tiles an SM: M = 768 78k 103 / 206, 234k 290 / 287, 469k 564
//   / 451, 1.6M 1925 / 1530; M = 896 200k 285 / 331, 402k 552 / 462; M = 640 281k
//   297 / 253, 560k 583 / 453.
//   32 columns, three (M < 600): M = 512 1.2M 764 / 772, 2.3M 1614 / 1493; M = 576
//   1.0M 743 / 773, 2.1M 1601 / 1509; M = 460 1.3M 767 / 832, 2.6M 1618 / 1524
//   (one state 1.7M 1138 / 1000); M = 597 1.0M 609 / 732.
//   64 columns: M = 440 2.7M 1418 / 1506; M = 257 4.7M 1399 / 1510.
bool stream_replicas(int M, int64_t n, int n_sel) {
    const int log2_p = sync_tile_log2_p(M);
    const int64_t columns = n * n_sel;
    if (log2_p >= 4) return false;
    if (log2_p <= 2) return columns >= 200000;
    return columns >= (M < 600 ? 1400000 : 300000);
}

// Deterministic block sum of one double per thread; result valid in thread 0.
__device__ double block_sum(double v) {
    __shared__ double part[kNormThreads / 32];
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) part[w] = v;
    __syncthreads();
    double total = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < static_cast<int>(blockDim.x >> 5); ++i) total += part[i];
    return total;
}

// A position of the norm kernels is one 16-byte load of the gradient: 4 f32
// or 8 bf16 values (8-byte bf16 loads, half the bytes per load instruction,
// read the ~350M workload's gradients at 5.56 TB/s).  A thread loads
// kNormUnroll positions before it accumulates them: i, i + T, ...,
// i + (U - 1) T with T the replica's thread count, the same order as a
// plain grid-stride loop, so the sums do not depend on the unrolling.
// 64 bytes per thread in flight.
constexpr int kNormUnroll = 4;

template <int GDT>
struct NormPos;
template <>
struct NormPos<MTDAO_F32> {
    static constexpr int E = 4;
    using W = float4;
};
template <>
struct NormPos<MTDAO_BF16> {
    static constexpr int E = 8;
    using W = uint4;
};

template <int GDT>
__device__ __forceinline__ typename NormPos<GDT>::W ld_grad_words(const void *g, int64_t e) {
    if constexpr (GDT == MTDAO_F32)
        return __ldcs(reinterpret_cast<const float4 *>(static_cast<const float *>(g) + e));
    else
        return __ldcs(reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(g) + e));
}

// The position's values in fp32 (bf16 -> fp32 is exact: the bits move up by 16).
template <int GDT>
__device__ __forceinline__ void widen(const typename NormPos<GDT>::W &w, float (&q)[NormPos<GDT>::E]) {
    if constexpr (GDT == MTDAO_F32) {
        q[0] = w.x; q[1] = w.y; q[2] = w.z; q[3] = w.w;
    } else {
        const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            q[2 * k] = __uint_as_float(u[k] << 16);
            q[2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u);
        }
    }
}

// fp32 range of a position's sum of four squares that the Kahan sum takes:
// above kSqHi a square or the sum may overflow (|g| above ~1.8e19 squares to
// Inf in fp32), below kSqLo a square may have lost bits to underflow (|g|
// below ~1e-19).  Positions outside it (and NaN / Inf) are summed in fp64
// instead, where every finite fp32 value squares exactly enough; the all-zero
// positions of padding and unused rows stay on the fp32 path.  A replica has
// at least 256 threads and, to fit in device memory, fewer than 2^34
// elements, so a thread adds fewer than 2^24 positions of at most 2^100:
// the fp32 sum stays finite.
constexpr float kSqHi = 0x1p100f;
constexpr float kSqLo = 0x1p-100f;

template <int GDT>
__global__ void __launch_bounds__(kNormThreads, 4) sqnorm_partial_kernel(const void *g, int64_t n,
                                                                      double *partial) {
    constexpr int E = NormPos<GDT>::E;
    const int m = blockIdx.y;
    const int nb = gridDim.x;
    const int64_t np = n / E;
    const int64_t T = static_cast<int64_t>(nb) * blockDim.x;
    float sum = 0.0f, comp = 0.0f;
    double wide = 0.0;                 // positions outside [kSqLo, kSqHi]
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < np;
         i += kNormUnroll * T) {
        typename NormPos<GDT>::W w[kNormUnroll];
#pragma unroll
        for (int u = 0; u < kNormUnroll; ++u)
            if (i + u * T < np) w[u] = ld_grad_words<GDT>(g, m * n + E * (i + u * T));
#pragma unroll
        for (int u = 0; u < kNormUnroll; ++u) {
            if (i + u * T >= np) break;
            float q[E];
            widen<GDT>(w[u], q);
            float p = __fmul_rn(q[E - 1], q[E - 1]);
            uint32_t bits = __float_as_uint(q[E - 1]);
#pragma unroll
            for (int k = E - 2; k >= 0; --k) {
                p = fmaf(q[k], q[k], p);
                bits |= __float_as_uint(q[k]);
            }
            const bool tiny = p < kSqLo && (bits & 0x7fffffffu) != 0u;
            if (!(p <= kSqHi) || tiny) {
                double d = static_cast<double>(q[E - 1]) * q[E - 1];
#pragma unroll
                for (int k = E - 2; k >= 0; --k) d = fma(static_cast<double>(q[k]), static_cast<double>(q[k]), d);
                wide += d;
                continue;
            }
            const float y = p - comp;
            const float t = sum + y;
            comp = (t - sum) - y;
            sum = t;
        }
    }
    const double total = block_sum((static_cast<double>(sum) - static_cast<double>(comp)) + wide);
    if (threadIdx.x == 0) partial[static_cast<int64_t>(m) * nb + blockIdx.x] = total;
}

// Number of NaN or +-Inf values (all exponent bits set) per replica, with
// the same fixed grid and reduction order as the sum of squares; counts are
// integers well below 2^53, so the double partials are exact.
template <int GDT>
__global__ void __launch_bounds__(kNormThreads, 4) nonfinite_partial_kernel(const void *g, int64_t n,
                                                                         double *partial) {
    constexpr int E = NormPos<GDT>::E;
    const int m = blockIdx.y;
    const int nb = gridDim.x;
    const int64_t np = n / E;
    const int64_t T = static_cast<int64_t>(nb) * blockDim.x;
    const uint32_t ex = 0x7f800000u;
    uint32_t count = 0;                // at most E np / T per thread
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < np;
         i += kNormUnroll * T) {
        typename NormPos<GDT>::W w[kNormUnroll];
#pragma unroll
        for (int u = 0; u < kNormUnroll; ++u)
            if (i + u * T < np) w[u] = ld_grad_words<GDT>(g, m * n + E * (i + u * T));
#pragma unroll
        for (int u = 0; u < kNormUnroll; ++u) {
            if (i + u * T >= np) break;
            float q[E];
            widen<GDT>(w[u], q);
#pragma unroll
            for (int k = 0; k < E; ++k) count += (__float_as_uint(q[k]) & ex) == ex;
        }
    }
    const double total = block_sum(static_cast<double>(count));
    if (threadIdx.x == 0) partial[static_cast<int64_t>(m) * nb + blockIdx.x] = total;
}

__global__ void __launch_bounds__(kNormThreads) sqnorm_finalize_kernel(const double *partial, int nb,
                                                                       double *out, float *clip_scale,
                                                                       double rho) {
    const int m = blockIdx.x;
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += partial[static_cast<int64_t>(m) * nb + i];
    const double total = block_sum(acc);
    if (threadIdx.x == 0) {
        out[m] = total;
        if (clip_scale != nullptr) {
            const double f = rho / (sqrt(total) + 1e-6);
            clip_scale[m] = static_cast<float>(f < 1.0 ? f : 1.0);
        }
    }
}

// ---------------------------------------------------------------- sync + diagnostics

// The block's sums of Q values per thread, value j to out[j * stride].
template <int Q>
__device__ __forceinline__ void block_sums(const Kahan (&acc)[Q], double *out, int64_t stride) {
    __shared__ double part[Q][kThreads / 32];
    int j;
    bool one;
    const double sum = warp_sums_wide<Q>(acc, j, one);
    if (one) part[j][threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x < Q) {
        double total = 0.0;
        for (int i = 0; i < kThreads / 32; ++i) total += part[threadIdx.x][i];
        out[threadIdx.x * stride] = total;
    }
}

// Replica average of the selected states (exactly as sync_kernel) plus, in
// the same pass over the M replicas, per state and block the partial sums of
//   q = 0          sum_m (s_m - s_bar)^2        (cross-worker variance * M)
//   q = 1          s_bar^2
//   q = 2 + m      s_m^2
//   q = 2 + M + m  s_m * s_bar
// written to partial[(sel * Q + q) * gridDim.x + block], Q = 2 + 2M.  s_bar
// is the fp32 mean that is stored, to the state's anchor too where it has one
// (a copy of replica 0 after the pass took 176 us of the ~124M list's 2942 at
// a round's end).  With M = 1 nothing is stored (there is nothing to average)
// but the sums are still formed.
template <int M>
__global__ void __launch_bounds__(kThreads) sync_stats_kernel(const __grid_constant__ SyncArgs a, int tile, double *partial) {
    constexpr int Q = 2 + 2 * M;
    float *base = a.arena + static_cast<int64_t>(a.sel[blockIdx.y]) * a.stride;
    const int64_t n = a.n_padded;
    const int64_t nv = n / 4;
    Kahan acc[Q];
    const int64_t first = static_cast<int64_t>(blockIdx.x) * tile * blockDim.x + threadIdx.x;
    for (int k = 0; k < tile; ++k) {
        const int64_t i = first + static_cast<int64_t>(k) * blockDim.x;
        if (i >= nv) break;
        const int64_t e = 4 * i;
        float r[M][4];
#pragma unroll
        for (int m = 0; m < M; ++m) to_array(ld_state(base + m * n + e), r[m]);
        float mean[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) mean[k] = replica_mean<M>([&](int m) { return r[m][k]; });
        float q[Q];
#pragma unroll
        for (int j = 0; j < Q; ++j) q[j] = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            q[1] = fmaf(mean[k], mean[k], q[1]);
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const float dv = r[m][k] - mean[k];
                q[0] = fmaf(dv, dv, q[0]);
                q[2 + m] = fmaf(r[m][k], r[m][k], q[2 + m]);
                q[2 + M + m] = fmaf(r[m][k], mean[k], q[2 + M + m]);
            }
        }
#pragma unroll
        for (int j = 0; j < Q; ++j) acc[j].add(q[j]);
        if constexpr (M > 1) {
            const float4 mv = from_array(mean);
#pragma unroll
            for (int m = 0; m < M; ++m) st_state(base + m * n + e, mv);
            if (a.anchor[blockIdx.y] != nullptr) st_state(a.anchor[blockIdx.y] + e, mv);
        }
    }
    block_sums<Q>(acc, partial + static_cast<int64_t>(blockIdx.y) * Q * gridDim.x + blockIdx.x, gridDim.x);
}

// stats[row * Q + q] = the sum over blocks of partial[(row * Q + q) * blocks + b]
// in fp64, WARPS warps a sum: thread t of them adds blocks t, t + 32 WARPS, ... in
// order, then the lanes and the warps are added in a fixed order.  q = 0 is divided
// by divide_first (M for the variance, a mean over workers; 0 leaves it).
template <int WARPS>
__global__ void __launch_bounds__(kNormThreads) stats_finalize_kernel(const double *partial, int64_t blocks, int Q,
                                                                      int n_sums, int divide_first, double *stats) {
    const int sum = WARPS == 1 ? static_cast<int>((blockIdx.x * kNormThreads + threadIdx.x) >> 5) : blockIdx.x;
    const int t = WARPS == 1 ? threadIdx.x & 31 : threadIdx.x;
    if (sum >= n_sums) return;
    const double *p = partial + static_cast<int64_t>(sum) * blocks;
    double acc = 0.0;
#pragma unroll 4
    for (int64_t b = t; b < blocks; b += 32 * WARPS) acc += p[b];
    const double total = WARPS == 1 ? warp_sum(acc) : block_sum(acc);
    if (t == 0) stats[sum] = (divide_first > 0 && sum % Q == 0) ? total / divide_first : total;
}

// A block for each sum, or a warp where there are many sums of few blocks: adding
// the lanes and warps of a block is 48 fp64 instructions, 16 cycles of the SM each,
// against blocks / 32 (average with sums, us, a block / a warp each, in brackets
// sums and blocks: M = 1024, n = 1219, 5 states (10250, 160) 73 / 46; M = 200, n =
// 30k, 3 states (1206, 473) 40.6 / 37.7; M = 64, n = 300, 5 states (650, 40) 7.6 /
// 6.3; but n = 286k, 4 states (520, 559) 112 / 114).
cudaError_t launch_finalize(const double *partial, int64_t blocks, int Q, int rows, int divide_first, double *stats,
                            cudaStream_t stream) {
    const int n_sums = Q * rows;
    if (n_sums >= 256 && blocks <= (n_sums >= 1024 ? 1024 : 256))
        stats_finalize_kernel<1><<<(n_sums + 7) / 8, kNormThreads, 0, stream>>>(partial, blocks, Q, n_sums,
                                                                               divide_first, stats);
    else
        stats_finalize_kernel<kNormThreads / 32><<<n_sums, kNormThreads, 0, stream>>>(partial, blocks, Q, n_sums,
                                                                                     divide_first, stats);
    return cudaGetLastError();
}

int64_t stats_blocks(int64_t n_padded, int tile) {
    const int64_t nv = n_padded / 4;
    const int64_t per_block = static_cast<int64_t>(tile) * kThreads;
    const int64_t b = (nv + per_block - 1) / per_block;
    return b < 1 ? 1 : b;
}

// Float4 positions a thread of sync_stats_kernel takes, consecutive for its
// block: block b covers positions [b * tile * 256, (b + 1) * tile * 256) of a
// state.  One block per tile, started in index order as earlier blocks retire;
// every block leaves one row of sums for stats_finalize_kernel, so the sums
// do not depend on the SM count.  A short tile keeps the addresses under way
// close together; what it pays for is the row at its end (2M + 2 sums over the
// block: as pairs within a warp, in fp64 from there on).  The average of 4
// states with its sums, us, tiles of 128 with every sum in fp64 -> of 16, here
// (in brackets 4, 8, 32, 128): M = 1, n = 60M 340 -> 312 (361, 327, 303, 326);
// M = 2 803 -> 610 (627, 610, 613, 654); M = 4 1362 -> 1168 (1155, 1169, 1178,
// 1234; 6.6 TB/s); M = 8, n = 30M 1307 -> 1159 (1167, 1169, 1186, 1213).  The
// warps' sums in fp64 too took 1178 (M = 4), 661 where this takes 614 (M = 6,
// n = 20M) and 48 where this takes 20 (M = 4, n = 1M).  Smaller states take
// shorter tiles, down to two positions, for 256 blocks: M = 4, n = 1M 98 -> 20,
// n = 100k 66 -> 6.5.
int sync_stats_tile(int64_t n_padded) {
    int tile = 16;
    while (tile > 2 && stats_blocks(n_padded, tile) < 256) tile /= 2;
    return tile;
}

template <int M>
cudaError_t launch_sync_stats_t(const SyncArgs &a, double *partial, size_t partial_cap, double *stats,
                                cudaStream_t stream) {
    constexpr int Q = 2 + 2 * M;
    const int tile = sync_stats_tile(a.n_padded);
    const int64_t gx = stats_blocks(a.n_padded, tile);
    if (static_cast<size_t>(gx) * a.n_sel * Q > partial_cap || gx > 0x7fffffff) return cudaErrorInvalidValue;
    dim3 grid(static_cast<unsigned>(gx), static_cast<unsigned>(a.n_sel));
    sync_stats_kernel<M><<<grid, kThreads, 0, stream>>>(a, tile, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_finalize(partial, gx, Q, a.n_sel, M, stats, stream);
}

// Pseudo-gradient diagnostics of the parameters x[M][n] against the anchor
// a[n] (the parameters at the last average), read-only, on a persistent
// grid, with fixed-order sums into partial[q * gridDim.x + block], Q = 2M + 2:
//   q = m          (x_m - a)^2
//   q = M + m      (x_m - a) * (x_bar - a)
//   q = 2M         (x_bar - a)^2
//   q = 2M + 1     a^2
// x_bar is the replica mean of replica_mean.cuh (the value an average would
// store now).  Blocks in index order with 16 positions a thread, as the sync
// diagnostics have them, took 186 us where this takes 176 (M = 4, n = 60M: 6.8
// TB/s; 197 with fp64 rows).
template <int M>
__global__ void __launch_bounds__(kThreads) pseudo_grad_stats_kernel(const float *x, const float *anchor,
                                                                     int64_t n, double *partial) {
    constexpr int Q = 2 * M + 2;
    const int64_t nv = n / 4;
    Kahan acc[Q];
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nv;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t e = 4 * i;
        float r[M][4], av[4];
#pragma unroll
        for (int m = 0; m < M; ++m) to_array(ld_state(x + m * n + e), r[m]);
        to_array(__ldcs(reinterpret_cast<const float4 *>(anchor + e)), av);
        float q[Q];
#pragma unroll
        for (int j = 0; j < Q; ++j) q[j] = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float mean = replica_mean<M>([&](int m) { return r[m][k]; });
            const float glob = mean - av[k];
            q[2 * M] = fmaf(glob, glob, q[2 * M]);
            q[2 * M + 1] = fmaf(av[k], av[k], q[2 * M + 1]);
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const float loc = r[m][k] - av[k];
                q[m] = fmaf(loc, loc, q[m]);
                q[M + m] = fmaf(loc, glob, q[M + m]);
            }
        }
#pragma unroll
        for (int j = 0; j < Q; ++j) acc[j].add(q[j]);
    }
    block_sums<Q>(acc, partial + blockIdx.x, gridDim.x);
}

template <int M>
cudaError_t launch_pseudo_grad_stats_t(const float *x, const float *anchor, int64_t n, int num_sms,
                                       double *partial, size_t partial_cap, double *stats,
                                       cudaStream_t stream) {
    constexpr int Q = 2 * M + 2;
    static const int per_sm = blocks_per_sm(pseudo_grad_stats_kernel<M>);
    int64_t gx = static_cast<int64_t>(per_sm) * num_sms;
    const int64_t need = (n / 4 + kThreads - 1) / kThreads;
    if (gx > need) gx = need;
    if (gx < 1) gx = 1;
    if (static_cast<size_t>(gx) * Q > partial_cap) return cudaErrorInvalidValue;
    pseudo_grad_stats_kernel<M><<<static_cast<unsigned>(gx), kThreads, 0, stream>>>(x, anchor, n, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the same fixed-order finalisation as the sync diagnostics, with no division
    return launch_finalize(partial, gx, Q, 1, 0, stats, stream);
}

// ---------------------------------------------------------------- diagnostics, replicas streamed

// For many replicas of large states (stream_stats) the diagnostics take two
// passes over a state; a [n] fp32 scratch holds the mean between them:
//   pass 1 (grid-stride over float4 positions): the replica mean of
//     replica_mean.cuh, written to the scratch (and to the state's anchor),
//     and the sums that need only the mean (and the anchor);
//   pass 2 (grid (blocks, M)): per replica the sums against the scratch mean
//     and, for an average, the mean written over the replica.
// The sums go as in the one-pass kernels: four elements in fp32, a thread's
// positions with Kahan compensation, warps, blocks and the finalize in fp64.

// Positions a pass-2 thread loads before it accumulates them (i, i + T,
// i + 2T, ...: the order of a plain grid-stride loop): four for the sync
// diagnostics (two float4 loads per position), two for the change
// diagnostics (three per position, within 64 registers).
constexpr int kPass2Unroll = 4;
constexpr int kPass2UnrollChange = 2;

// Pass 1.  Per block s_bar^2, or with CHANGE (x_bar - a)^2 and a^2: value j at
// partial[j * gridDim.x + block].
template <bool CHANGE>
__global__ void __launch_bounds__(kThreads, 4) stream_stats_pass1_kernel(const float *s, const float *anchor, int64_t n,
                                                                         int M, float *mean_out, float *new_anchor,
                                                                         double *partial) {
    constexpr int K = CHANGE ? 2 : 1;
    const int64_t nv = n / 4;
    Kahan acc[K];
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nv;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t e = 4 * i;
        const float4 mv = replica_mean4(s, n, M, e);
        *reinterpret_cast<float4 *>(mean_out + e) = mv;
        if (new_anchor != nullptr) st_state(new_anchor + e, mv);
        float mean[4], p0 = 0.0f;
        to_array(mv, mean);
        if constexpr (CHANGE) {
            float a[4], p1 = 0.0f;
            to_array(__ldcs(reinterpret_cast<const float4 *>(anchor + e)), a);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float glob = mean[k] - a[k];
                p0 = fmaf(glob, glob, p0);
                p1 = fmaf(a[k], a[k], p1);
            }
            acc[K - 1].add(p1);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) p0 = fmaf(mean[k], mean[k], p0);
        }
        acc[0].add(p0);
    }
    block_sums<K>(acc, partial + blockIdx.x, gridDim.x);
}

// Pass 2 of the sync diagnostics, replica m = blockIdx.y: per block
// (s_m - s_bar)^2, s_m^2 and s_m * s_bar, value j at
// partial[(j * M + m) * gridDim.x + block]; the replica becomes the mean.
__global__ void __launch_bounds__(kThreads, 4) stream_sync_stats_pass2_kernel(float *s, int64_t n, const float *mean,
                                                                              double *partial) {
    const int m = blockIdx.y;
    const int64_t nv = n / 4;
    const int64_t T = static_cast<int64_t>(gridDim.x) * blockDim.x;
    float *rep = s + m * n;
    Kahan acc[3];
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nv; i += kPass2Unroll * T) {
        float4 rv[kPass2Unroll], mv[kPass2Unroll];
#pragma unroll
        for (int u = 0; u < kPass2Unroll; ++u)
            if (i + u * T < nv) {
                rv[u] = ld_state(rep + 4 * (i + u * T));
                mv[u] = *reinterpret_cast<const float4 *>(mean + 4 * (i + u * T));
            }
#pragma unroll
        for (int u = 0; u < kPass2Unroll; ++u) {
            if (i + u * T >= nv) break;
            float r[4], mb[4];
            to_array(rv[u], r);
            to_array(mv[u], mb);
            float p0 = 0.0f, p1 = 0.0f, p2 = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float dv = r[k] - mb[k];
                p0 = fmaf(dv, dv, p0);
                p1 = fmaf(r[k], r[k], p1);
                p2 = fmaf(r[k], mb[k], p2);
            }
            acc[0].add(p0);
            acc[1].add(p1);
            acc[2].add(p2);
            st_state(rep + 4 * (i + u * T), mv[u]);
        }
    }
    block_sums<3>(acc, partial + static_cast<int64_t>(m) * gridDim.x + blockIdx.x,
                  static_cast<int64_t>(gridDim.y) * gridDim.x);
}

// Pass 2 of the change diagnostics, replica m = blockIdx.y: per block
// (x_m - a)^2 and (x_m - a)(x_bar - a), laid out as above.  Read-only.
__global__ void __launch_bounds__(kThreads, 4) stream_change_pass2_kernel(const float *x, const float *anchor, int64_t n,
                                                                          const float *mean, double *partial) {
    const int m = blockIdx.y;
    const int64_t nv = n / 4;
    const int64_t T = static_cast<int64_t>(gridDim.x) * blockDim.x;
    const float *rep = x + m * n;
    Kahan acc[2];
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nv; i += kPass2UnrollChange * T) {
        float4 rv[kPass2UnrollChange], mv[kPass2UnrollChange], av[kPass2UnrollChange];
#pragma unroll
        for (int u = 0; u < kPass2UnrollChange; ++u)
            if (i + u * T < nv) {
                const int64_t e = 4 * (i + u * T);
                rv[u] = ld_state(rep + e);
                mv[u] = *reinterpret_cast<const float4 *>(mean + e);
                av[u] = *reinterpret_cast<const float4 *>(anchor + e);
            }
#pragma unroll
        for (int u = 0; u < kPass2UnrollChange; ++u) {
            if (i + u * T >= nv) break;
            float r[4], mb[4], a[4];
            to_array(rv[u], r);
            to_array(mv[u], mb);
            to_array(av[u], a);
            float p0 = 0.0f, p1 = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float loc = r[k] - a[k];
                const float glob = mb[k] - a[k];
                p0 = fmaf(loc, loc, p0);
                p1 = fmaf(loc, glob, p1);
            }
            acc[0].add(p0);
            acc[1].add(p1);
        }
    }
    block_sums<2>(acc, partial + static_cast<int64_t>(m) * gridDim.x + blockIdx.x,
                  static_cast<int64_t>(gridDim.y) * gridDim.x);
}

struct StreamGrid {
    int b1, b2;                      // blocks of pass 1, and of a replica in pass 2
};

StreamGrid stream_grid2(int num_sms, int M, int64_t n) {
    const int64_t need = (n / 4 + kThreads - 1) / kThreads;
    int64_t b1 = 4 * static_cast<int64_t>(num_sms), b2 = b1 / M;
    if (b1 > need) b1 = need;
    if (b2 > need) b2 = need;
    return {static_cast<int>(b1 < 1 ? 1 : b1), static_cast<int>(b2 < 1 ? 1 : b2)};
}

}  // namespace

// Two passes with rows of 512 bytes a warp against one pass on tiles of 32 or 16
// columns.  us, tiles / streamed:
//   16 columns (M > 898): M = 1024, average with sums of one state n = 59k 257 /
//   316, 117k 471 / 404, 391k 1514 / 848; change n = 59k 226 / 279, 117k 409 /
//   326, 781k 2413 / 1159.
//   32 columns: change M = 512 234k 206 / 220, 391k 325 / 294, 1.6M 1162 / 1060; M
//   = 600 267k 349 / 260, M = 768 156k 268 / 297, 260k 399 / 382, 1.0M 1384 / 1230; average with sums M = 896 223k 490 /
//   518, 446k 1025 / 854; M = 768 521k 994 / 862; M = 640 312k 532 / 482, three
//   states 1472 / 1441.  Up to M = 598 three tiles fit an SM: M = 512 781k 821 /
//   921.
//   M < 450 (32 columns from M = 257, 64 below): M = 440 change 1.8M 996 / 1102.
bool stream_stats(int M, int64_t n, bool change) {
    if (M < 450) return false;
    if (M > 898) return n >= (change ? 81920 : 98304);
    return change ? n >= (M < 599 ? 262144 : 196608) : M >= 599 && n >= 393216;
}

size_t stream_stats_partial_capacity(int num_sms, int64_t n_padded, int M) {
    const StreamGrid g = stream_grid2(num_sms, M, n_padded);
    return 2 * static_cast<size_t>(g.b1) + 3 * static_cast<size_t>(g.b2) * static_cast<size_t>(M);
}

cudaError_t launch_sync_stats_stream(const SyncArgs &a, int num_sms, float *mean, double *partial, size_t partial_cap,
                                     double *stats, cudaStream_t stream) {
    const int M = a.M;
    const StreamGrid g = stream_grid2(num_sms, M, a.n_padded);
    if (stream_stats_partial_capacity(num_sms, a.n_padded, M) > partial_cap) return cudaErrorInvalidValue;
    double *p1 = partial, *p2 = partial + g.b1;
    const int64_t per_sum = static_cast<int64_t>(M) * g.b2;
    for (int k = 0; k < a.n_sel; ++k, stats += 2 + 2 * M) {
        float *s = a.arena + static_cast<int64_t>(a.sel[k]) * a.stride;
        stream_stats_pass1_kernel<false><<<g.b1, kThreads, 0, stream>>>(s, nullptr, a.n_padded, M, mean, a.anchor[k], p1);
        stream_sync_stats_pass2_kernel<<<dim3(g.b2, M), kThreads, 0, stream>>>(s, a.n_padded, mean, p2);
        // stats row: [0] variance (over all replicas' blocks), [1] s_bar^2, [2 + m] s_m^2, [2 + M + m] s_m s_bar
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess) e = launch_finalize(p2, per_sum, 1, 1, M, stats, stream);
        if (e == cudaSuccess) e = launch_finalize(p1, g.b1, 1, 1, 0, stats + 1, stream);
        if (e == cudaSuccess) e = launch_finalize(p2 + per_sum, g.b2, 2 * M, 1, 0, stats + 2, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_pseudo_grad_stats_stream(const float *x, const float *anchor, int64_t n, int M, int num_sms,
                                            float *mean, double *partial, size_t partial_cap, double *stats,
                                            cudaStream_t stream) {
    const StreamGrid g = stream_grid2(num_sms, M, n);
    if (stream_stats_partial_capacity(num_sms, n, M) > partial_cap) return cudaErrorInvalidValue;
    double *p1 = partial, *p2 = partial + 2 * g.b1;
    stream_stats_pass1_kernel<true><<<g.b1, kThreads, 0, stream>>>(x, anchor, n, M, mean, nullptr, p1);
    stream_change_pass2_kernel<<<dim3(g.b2, M), kThreads, 0, stream>>>(x, anchor, n, mean, p2);
    // [m] (x_m - a)^2, [M + m] (x_m - a)(x_bar - a), [2M] (x_bar - a)^2, [2M + 1] a^2
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_finalize(p2, g.b2, 2 * M, 1, 0, stats, stream);
    if (e == cudaSuccess) e = launch_finalize(p1, g.b1, 2, 1, 0, stats + 2 * M, stream);
    return e;
}

cudaError_t launch_pseudo_grad_stats(const float *x, const float *anchor, int64_t n, int M, int num_sms,
                                     double *partial, size_t partial_cap, double *stats,
                                     cudaStream_t stream) {
    switch (M) {
        case 1: return launch_pseudo_grad_stats_t<1>(x, anchor, n, num_sms, partial, partial_cap, stats, stream);
        case 2: return launch_pseudo_grad_stats_t<2>(x, anchor, n, num_sms, partial, partial_cap, stats, stream);
        case 3: return launch_pseudo_grad_stats_t<3>(x, anchor, n, num_sms, partial, partial_cap, stats, stream);
        case 4: return launch_pseudo_grad_stats_t<4>(x, anchor, n, num_sms, partial, partial_cap, stats, stream);
        case 5: return launch_pseudo_grad_stats_t<5>(x, anchor, n, num_sms, partial, partial_cap, stats, stream);
        case 6: return launch_pseudo_grad_stats_t<6>(x, anchor, n, num_sms, partial, partial_cap, stats, stream);
        case 7: return launch_pseudo_grad_stats_t<7>(x, anchor, n, num_sms, partial, partial_cap, stats, stream);
        case 8: return launch_pseudo_grad_stats_t<8>(x, anchor, n, num_sms, partial, partial_cap, stats, stream);
        default: return cudaErrorNotSupported;
    }
}

size_t sync_stats_partial_capacity(int num_sms, int64_t n_padded, int n_states, int M) {
    // one row of 2 + 2M sums per block and state, or per persistent block
    // of the pseudo-gradient pass (at most 16 resident blocks per SM)
    const size_t sync = static_cast<size_t>(stats_blocks(n_padded, sync_stats_tile(n_padded))) * n_states;
    const size_t change = static_cast<size_t>(16) * num_sms;
    return (sync > change ? sync : change) * (2 + 2 * static_cast<size_t>(M));
}

cudaError_t launch_sync_stats(const SyncArgs &a, int num_sms, double *partial, size_t partial_cap,
                              double *stats, cudaStream_t stream) {
    if (a.n_sel <= 0) return cudaSuccess;
    switch (a.M) {
        case 1: return launch_sync_stats_t<1>(a, partial, partial_cap, stats, stream);
        case 2: return launch_sync_stats_t<2>(a, partial, partial_cap, stats, stream);
        case 3: return launch_sync_stats_t<3>(a, partial, partial_cap, stats, stream);
        case 4: return launch_sync_stats_t<4>(a, partial, partial_cap, stats, stream);
        case 5: return launch_sync_stats_t<5>(a, partial, partial_cap, stats, stream);
        case 6: return launch_sync_stats_t<6>(a, partial, partial_cap, stats, stream);
        case 7: return launch_sync_stats_t<7>(a, partial, partial_cap, stats, stream);
        case 8: return launch_sync_stats_t<8>(a, partial, partial_cap, stats, stream);
        default: return cudaErrorNotSupported;
    }
}

cudaError_t launch_sync(const SyncArgs &a, int num_sms, cudaStream_t stream) {
    if (a.n_sel <= 0 || a.M <= 1) return cudaSuccess;
    switch (a.M) {
        case 2: return launch_sync_t<2>(a, stream);
        case 3: return launch_sync_t<3>(a, stream);
        case 4: return launch_sync_t<4>(a, stream);
        case 5: return launch_sync_t<5>(a, stream);
        case 6: return launch_sync_t<6>(a, stream);
        case 7: return launch_sync_t<7>(a, stream);
        case 8: return launch_sync_t<8>(a, stream);
        case 9: return launch_sync_t<9>(a, stream);
        case 10: return launch_sync_t<10>(a, stream);
        case 11: return launch_sync_t<11>(a, stream);
        case 12: return launch_sync_t<12>(a, stream);
        case 13: return launch_sync_t<13>(a, stream);
        case 14: return launch_sync_t<14>(a, stream);
        default:
            return stream_replicas(a.M, a.n_padded, a.n_sel) ? launch_sync_stream(a, num_sms, stream)
                                                             : launch_sync_tile(a, num_sms, stream);
    }
}

int norm_blocks_per_replica(int num_sms, int M) {
    int b = (4 * num_sms) / (M > 0 ? M : 1);
    return b < 1 ? 1 : b;
}

cudaError_t launch_grad_nonfinite(const void *grads, int grad_dtype, int32_t M, int64_t n_padded,
                                  int blocks_per_replica, double *partial, double *out, cudaStream_t stream) {
    dim3 grid(static_cast<unsigned>(blocks_per_replica), static_cast<unsigned>(M));
    if (grad_dtype == MTDAO_F32)
        nonfinite_partial_kernel<MTDAO_F32><<<grid, kNormThreads, 0, stream>>>(grads, n_padded, partial);
    else
        nonfinite_partial_kernel<MTDAO_BF16><<<grid, kNormThreads, 0, stream>>>(grads, n_padded, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sqnorm_finalize_kernel<<<M, kNormThreads, 0, stream>>>(partial, blocks_per_replica, out, nullptr, 0.0);
    return cudaGetLastError();
}

cudaError_t launch_grad_sqnorm(const void *grads, int grad_dtype, int32_t M, int64_t n_padded,
                               int blocks_per_replica, double *partial, double *out,
                               float *clip_scale, double rho, cudaStream_t stream) {
    dim3 grid(static_cast<unsigned>(blocks_per_replica), static_cast<unsigned>(M));
    if (grad_dtype == MTDAO_F32)
        sqnorm_partial_kernel<MTDAO_F32><<<grid, kNormThreads, 0, stream>>>(grads, n_padded, partial);
    else
        sqnorm_partial_kernel<MTDAO_BF16><<<grid, kNormThreads, 0, stream>>>(grads, n_padded, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sqnorm_finalize_kernel<<<M, kNormThreads, 0, stream>>>(partial, blocks_per_replica, out, clip_scale,
                                                          rho);
    return cudaGetLastError();
}


cudaError_t launch_stats_finalize(const double *partial, int64_t blocks, int Q, int rows, int divide_first,
                                  double *stats, cudaStream_t stream) {
    return launch_finalize(partial, blocks, Q, rows, divide_first, stats, stream);
}

}  // namespace mtdao
