// step_sync_wide.cuh -- the local step with the replica average fused in,
// for replica counts above what a lane holds (M = 9 to kTileMaxM) and for most
// of M = 3 to 8 on large states.
//
// A block owns a tile: S consecutive columns of all M replicas, of every
// state and of the gradient, copied to shared memory (cp.async) at once.
// Its threads update the tile with update_state; a state that is not due is
// stored from registers, a due state's new values go back over its tile.
// After one barrier the replica mean of every (due state, column) pair is
// formed (tile_means of replica_tile.cuh: the standalone average's sums in the
// same order, so fused and separate averaging give identical bits for every
// M); after a second barrier the means are stored to every replica.
//
// One tile per block, the blocks started in index order as earlier ones
// retire; what overlaps the copies of one block is the work of the others on
// its SM.  Against persistent blocks that copied their next span (of half
// the columns, for the same shared memory) while they worked on the current
// one: M = 16, n = 2^23, Adam N = 3, f32 5872 -> 6970 GB/s; M = 32 5706 ->
// 6850; M = 64, n = 1.9M, SGDM, bf16 4683 -> 6740; M = 100, n = 600k, Adam
// N = 2 (step and average apart before) 3423 -> 6120, M = 256 3406 -> 3871,
// SGDM 3384 -> 5340; M = 256, n = 512 63.5 -> 8.2 us.  Both halves count: a
// plain copy of such tiles runs at 6.7-6.9 TB/s with rows of 256 bytes or
// more in index order, 6.1-6.3 persistent, and 5.5-5.9 / 5.1-5.3 with rows of
// 128 bytes.  Bound by HBM up to M = 64; above, by the two or three blocks
// that fit on an SM (one where a tile takes more than 113 KB).
#pragma once

#include "replica_tile.cuh"
#include "step_kernels.cuh"

namespace mtdao {

constexpr int kTileMaxThreads = 512;      // largest block of the fused step
constexpr int kTileMaxM = 256;            // largest M of the fused step (above: step + average)

// Floats of one tile set: M x S floats per state and the gradient's
// (M x S f32, or bf16 in half the floats).
template <int BASE, int N, int GDT>
__host__ __device__ constexpr int tile_set_floats(int M, int S) {
    return kNumStates<BASE, N> * M * S + (GDT == MTDAO_F32 ? M * S : M * S / 2);
}

// Index of the k-th set bit of mask (k counts from 0 and is in range).
__device__ __forceinline__ int nth_set_bit(uint32_t mask, int k) {
    for (; k > 0; --k) mask &= mask - 1u;
    return __ffs(static_cast<int>(mask)) - 1;
}

// The fused step on one tile of S = 4 * 2^log2_p columns of all replicas per
// block.  Item i of the tile is float4 position i % 2^log2_p of replica
// i / 2^log2_p; a thread copies, updates and stores the same items (always the
// same position, as 2^log2_p divides the block), so the only barriers are those
// around the means.  A due state's updated values are written back over its
// own tile, a state that is not due goes straight to HBM.
template <int BASE, int N, int GDT, bool CLIP, int V>
__global__ void __launch_bounds__(kTileMaxThreads) step_sync_tile_kernel(const StepArgs a, int log2_p) {
    extern __shared__ __align__(16) float smem[];
    constexpr int kStates = kNumStates<BASE, N>;
    const int M = a.M;
    const int S = 4 << log2_p;
    const int tile = M * S;
    const int64_t n = a.n_padded;
    const int64_t stride = a.stride;
    const uint32_t mask = a.sync_mask;
    float *mean = smem + tile_set_floats<BASE, N, GDT>(M, S);   // [n_due][S]

    // The thread's items: replicas r, r + rows, ...; e: the element of item r.
    const int f = static_cast<int>(threadIdx.x) & ((1 << log2_p) - 1);
    const int r0 = static_cast<int>(threadIdx.x) >> log2_p;
    const int rows = static_cast<int>(blockDim.x) >> log2_p;
    const int64_t e0 = r0 * n + static_cast<int64_t>(blockIdx.x) * S + 4 * f;
    const int64_t e_step = rows * n;
    const int at0 = r0 * S + 4 * f, at_step = rows * S;          // in a tile

    {
        int64_t e = e0;
        int at = at0;
        for (int r = r0; r < M; r += rows, e += e_step, at += at_step) {
#pragma unroll
            for (int st = 0; st < kStates; ++st) cp_async16(smem + st * tile + at, a.arena + st * stride + e);
            if constexpr (GDT == MTDAO_F32)
                cp_async16(smem + kStates * tile + at, static_cast<const float *>(a.grads) + e);
            else
                cp_async8(reinterpret_cast<uint16_t *>(smem + kStates * tile) + at,
                          static_cast<const uint16_t *>(a.grads) + e);
        }
    }
    cp_async_commit();
    cp_async_wait<0>();                          // a thread reads what it copied itself

    {
        int64_t e = e0;
        int at = at0;
        for (int r = r0; r < M; r += rows, e += e_step, at += at_step) {
            const float s = CLIP ? __ldg(a.clip_scale + r) : 1.0f;
            float g[4], gt[4], acc[4];
            if constexpr (GDT == MTDAO_F32) {
                to_array(*reinterpret_cast<const float4 *>(smem + kStates * tile + at), g);
            } else {
                const uint2 w =
                    *reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(smem + kStates * tile) + at);
                g[0] = __uint_as_float(w.x << 16);
                g[1] = __uint_as_float(w.x & 0xffff0000u);
                g[2] = __uint_as_float(w.y << 16);
                g[3] = __uint_as_float(w.y & 0xffff0000u);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[k] = step_acc_init<BASE>(a.sc, g[k], s);
#pragma unroll
            for (int o = 0; o < kStates; ++o) {
                const int st = state_order<BASE, N>(o);
                float *cell = smem + st * tile + at;
                float cur[4];
                to_array(*reinterpret_cast<const float4 *>(cell), cur);
#pragma unroll
                for (int k = 0; k < 4; ++k) update_state<BASE, N>(a.sc, st, g[k], s, gt[k], acc[k], cur[k]);
                if ((mask >> st) & 1u)
                    *reinterpret_cast<float4 *>(cell) = from_array(cur);
                else
                    st_state(a.arena + st * stride + e, from_array(cur));
            }
        }
    }
    __syncthreads();
    tile_means<V>([=](int k) { return smem + nth_set_bit(mask, k) * tile; }, M, log2_p + 2, __popc(mask) * S, mean);
    __syncthreads();
    const float *from = mean + 4 * f;
#pragma unroll
    for (int st = 0; st < kStates; ++st) {
        if (((mask >> st) & 1u) == 0) continue;
        const float4 m4 = *reinterpret_cast<const float4 *>(from);
        from += S;
        float *to = a.arena + st * stride + e0;
        for (int r = r0; r < M; r += rows, to += e_step) st_state(to, m4);
    }
}

// Columns of a tile, threads of its block and the form of its means (tile_means'
// V).
struct TileShape {
    int S, threads, means;
    size_t smem;
};

// The shape for M replicas of n elements with n_due states due; bytes(S): the
// shared memory of a tile of S columns; sgdm_n_mom: SGDM's N (its update has no
// square root and division), else 0.
// Columns (fused step, GB/s): 128 up to M = 16 (M = 16, Adam N = 3: 6915, 64
// columns 5874, 256 5866), else 64 (M = 32: 6864, 128 columns 5970; M = 64, SGDM
// 6730, 128 columns 6541); 32 where two blocks of 64 would not fit an SM (M = 64,
// Adam N = 4: 5928, 64 columns 4583; M = 100, Adam N = 2: 5998, 16 columns
// 3711).  Small states, where rows count less (L2)
// and the SMs are to have tiles enough, take fewer: the half while an SM would
// get fewer tiles than tile_min of them (us: M = 16, n = 200k, ADOPT N = 3 128
// columns 27.8, 64 26.6; M = 47, n = 149k, ADOPT N = 2 64 columns 53.1, 32
// 48.1, 16 48.0; M = 64, n = 60k, Adam N = 2 28.7, 23.0, 23.8; M = 24, n = 500k
// 72.3, 71.8, 73.4; M = 44, n = 10k, ADOPT N = 3 11.3, 9.3, 8.2; M = 100, n =
// 4k 32 columns 8.2, 16 6.2, 8 8.2; M = 256, n = 512 32 columns 12.3, 8 8.2;
// M = 11, n = 111k, SGDM N = 4 128 columns 8.3, 32 11.8; M = 64, n = 1500, SGDM N
// = 1 and 3, ADOPT N = 4 16 columns 2.7, 3.1, 4.0, 8 2.9, 3.4, 4.3).
// Threads: about 1024 per SM over the blocks that fit, with 2 to 4 items each
// (M = 48, Adam N = 3: 3 items 6740, 2 items 6169; M = 9: 2 items 6508, 3
// items 6126, 1 item 4803); two items where that deals them out evenly to 256
// threads at most and the rule's count does not (M = 16, ADOPT, bf16: 2 items
// 6659, 3 items 6067).
// Means: four columns a lane where that still gives every lane one (us, one
// column -> four: M = 4, n = 20M, Adam N = 3 599 -> 514, ADOPT N = 2 488 -> 409; M
// = 6, ADOPT N = 2 741 -> 628; M = 12, n = 2^23 511 -> 496; but M = 8, ADOPT N =
// 2, three states due 785 -> 793, M = 16 659 -> 671).
// Up to 20 tiles an SM (states in L2) the other blocks do not hide a block's
// means, and their form is chosen by the columns due against the threads (M = 9 to
// 64; 19411 random steps of 250 elements to 30M over all replicas: 2.3 % faster in
// the mean, up to 16 %, and 6 % slower at most):
//   at most half as many columns, M >= 24 and tiles for few rounds (3 an SM, SGDM
//   6): a pair of half-warps (M = 56, n = 1500, SGDM N = 1 3.4 -> 2.75; M = 64, n =
//   5000 3.9 -> 3.15; but M = 32, n = 16k, Adam N = 2 4.55 -> 4.97);
//   more columns than threads, and fewer items a thread (two or more) give every
//   column a thread: those (M = 20, n = 130k, SGDM N = 1, 5 items 7.7, 3 7.1);
//   else twice as many columns, 256 or more: four a lane (M = 15, n = 130k, SGDM N =
//   3 12.7 -> 9.5; M = 17, n = 90k, 10.0 -> 8.6);
//   else M <= 16, SGDM N = 1: four a lane and 96 threads (M = 9, n = 130k 5.1 ->
//   4.4; M = 10, n = 180k 6.6 -> 5.9; with N >= 3 or more replicas it loses).
constexpr int64_t kTilesInL2 = 20;

template <typename Bytes>
TileShape tile_shape(int M, int64_t n, int num_sms, int n_due, int sgdm_n_mom, Bytes bytes) {
    TileShape w;
    w.S = M <= 16 ? 128 : 64;
    while (w.S > 32 && 2 * (bytes(w.S) + kSharedReserved) > kSharedPerSm) w.S /= 2;
    auto tile_min = [&](int S) {
        if (M * (S / 8) >= 256 && S >= 64) return S == 128 ? 11 : 16;      // the half still has items enough
        if (S >= 32) return 3;
        return S == 16 && M > 32 && M < kSplitMeansM ? 0 : 1;
    };
    while (w.S > 8 && (bytes(w.S) + kSharedReserved > kSharedPerSm || n / w.S < int64_t{num_sms} * tile_min(w.S)))
        w.S /= 2;
    w.smem = bytes(w.S);
    const int items = M * (w.S / 4);
    int64_t resident = (n / w.S + num_sms - 1) / num_sms;        // blocks of an SM
    if (resident > tile_blocks_fit(w.smem)) resident = tile_blocks_fit(w.smem);
    if (resident > 16) resident = 16;
    auto threads_of = [&](int per) {
        const int t = ((items + per - 1) / per + 31) / 32 * 32;
        return t < kTileMaxThreads ? t : kTileMaxThreads;
    };
    int per = static_cast<int>((items * resident + 1023) / 1024);    // items of a thread
    if (per > 2 && items % (32 * per) != 0 && items % 64 == 0 && items <= 512) per = 2;
    const int columns = n_due * w.S;
    const int64_t tiles = n / w.S;
    w.means = M >= kSplitMeansM ? 0 : (columns >= 4 * threads_of(per) ? 4 : 1);
    if (M >= 9 && M < kSplitMeansM && tiles < kTilesInL2 * num_sms) {
        if (2 * columns <= threads_of(per) && M >= 24 && tiles <= int64_t{num_sms} * (sgdm_n_mom > 0 ? 6 : 3)) {
            w.means = 0;
        } else if (columns > threads_of(per)) {
            int fewer = per - 1;
            while (fewer >= 2 && threads_of(fewer) < columns) --fewer;
            if (fewer >= 2) {
                per = fewer;
                w.means = 1;
            } else if (columns >= 256 && columns >= 2 * threads_of(per)) {
                w.means = 4;
            } else if (sgdm_n_mom == 1 && M <= 16 && w.means == 1) {
                if (per < (items + 95) / 96) per = (items + 95) / 96;
                w.means = 4;
            }
        }
    }
    w.threads = threads_of(per);
    return w;
}

template <int BASE, int N, int GDT, bool CLIP>
cudaError_t launch_step_sync_tile(const StepArgs &a, int num_sms, cudaStream_t stream) {
    if (a.M > kTileMaxM) return cudaErrorNotSupported;
    const int n_due = __builtin_popcount(a.sync_mask);
    const TileShape w = tile_shape(a.M, a.n_padded, num_sms, n_due, BASE == MTDAO_BASE_SGDM ? N : 0, [&](int S) {
        return (static_cast<size_t>(tile_set_floats<BASE, N, GDT>(a.M, S)) + static_cast<size_t>(n_due) * S) *
               sizeof(float);
    });
    // One tile an SM and one or two states due: the step and their average
    // apart (us, tiled / apart: M = 181, n = 300k, Adam N = 3, bf16, one state
    // due 469 / 395, three 503 / 520, five 581 / 645; M = 256, n = 150k, Adam N =
    // 4 364 / 338, 440 / 427, 496 / 515; with two tiles an SM M = 128, n = 500k,
    // Adam N = 2, one state due 381 / 404, M = 256 SGDM 340 / 417).
    if (tile_blocks_fit(w.smem) == 1 && n_due <= 2) return cudaErrorNotSupported;
    int log2_p = 0;
    while ((4 << log2_p) < w.S) ++log2_p;
    auto kernel = w.means == 0   ? step_sync_tile_kernel<BASE, N, GDT, CLIP, 0>
                  : w.means == 4 ? step_sync_tile_kernel<BASE, N, GDT, CLIP, 4>
                                 : step_sync_tile_kernel<BASE, N, GDT, CLIP, 1>;
    if (const cudaError_t e = allow_shared(kernel, w.smem); e != cudaSuccess) return e;
    kernel<<<static_cast<unsigned>(a.n_padded / w.S), w.threads, w.smem, stream>>>(a, log2_p);
    return cudaGetLastError();
}

}  // namespace mtdao
