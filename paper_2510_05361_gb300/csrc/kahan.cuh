// kahan.cuh -- the accumulators of the diagnostics and norm reductions.
#pragma once

#include <cuda_runtime.h>

namespace mtdao {

// fp32 accumulator with Kahan compensation; value() folds the compensation
// in at double precision.
struct Kahan {
    float s = 0.0f, c = 0.0f;
    __device__ __forceinline__ void add(float y) {
        y -= c;
        const float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const {
        return static_cast<double>(s) - static_cast<double>(c);
    }
};

// a + b, with a's and b's compensations: the rounding error of the sum joins
// them, so sums of such sums stay good to about 2^-46 of the sum of magnitudes
// (an fp64 instruction takes 16 cycles of the SM for one warp, this some seven
// of a quarter of it).  Not finite, as a double's would be, where the sum passes
// 3.4e38: the sums below then take fp64.
__device__ __forceinline__ Kahan operator+(const Kahan &a, const Kahan &b) {
    Kahan r;
    r.s = a.s + b.s;
    const float t = r.s - a.s;
    const float err = (a.s - (r.s - t)) + (b.s - t);   // a.s + b.s = r.s + err exactly
    r.c = (a.c + b.c) - err;
    return r;
}

__device__ __forceinline__ bool is_finite(const Kahan &v) { return fabsf(v.s) <= 3.402823466e38f; }

__device__ __forceinline__ double lane_xor(double v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
__device__ __forceinline__ Kahan lane_xor(const Kahan &v, int off) {
    Kahan r;
    r.s = __shfl_xor_sync(0xffffffffu, v.s, off);
    r.c = __shfl_xor_sync(0xffffffffu, v.c, off);
    return r;
}

// Sums of K values per lane over a warp, in a fixed order: the returned sum is
// that of value `at` of the K, in every lane (`one` is set in one lane of each).
// A step halves the values as well as the lanes that they are summed over (each
// lane hands the half that it does not keep to the other one): 12 additions for
// K = 10, 20 for K = 18, where a butterfly per value takes 5 K.
template <typename T, int K, int OFF = 16>
__device__ __forceinline__ T warp_sums(const T (&v)[K], int &at, bool &one) {
    if constexpr (OFF == 0) {
        at = 0;
        one = true;
        return v[0];
    } else {
        constexpr int H = (K + 1) / 2;
        const bool upper = (threadIdx.x & OFF) != 0;   // keeps values H .. K-1 (none for K = 1: a copy of the sum)
        T s[H];
        if constexpr (K == 1) {
            s[0] = v[0] + lane_xor(v[0], OFF);
        } else {
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const T high = H + i < K ? v[H + i < K ? H + i : 0] : T();
                s[i] = (upper ? high : v[i]) + lane_xor(upper ? v[i] : high, OFF);
            }
        }
        const T sum = warp_sums<T, H, OFF / 2>(s, at, one);
        if (upper) {
            at += H;
            one = one && at < K;
        }
        return sum;
    }
}

// The same for Kahan sums, in fp64: added as pairs, and where a sum is not
// finite that way as doubles.
template <int K>
__device__ __forceinline__ double warp_sums_wide(const Kahan (&v)[K], int &at, bool &one) {
    const Kahan sum = warp_sums<Kahan, K>(v, at, one);
    if (__all_sync(0xffffffffu, is_finite(sum))) return sum.value();
    double d[K];
#pragma unroll
    for (int j = 0; j < K; ++j) d[j] = v[j].value();
    return warp_sums<double, K>(d, at, one);
}

// Sums of two values over aligned groups of L lanes (a power of two from 2 to
// 32): a's in the even lanes, b's in the odd ones.  The whole warp calls it.
template <typename T>
__device__ __forceinline__ T lanes_sum2(const T &a, const T &b, int L) {
    const bool odd = (threadIdx.x & 1) != 0;
    T v = (odd ? b : a) + lane_xor(odd ? a : b, 1);
    for (int off = 2; off < L; off <<= 1) v = v + lane_xor(v, off);
    return v;
}
__device__ __forceinline__ double lanes_sum2_wide(const Kahan &a, const Kahan &b, int L) {
    const Kahan sum = lanes_sum2(a, b, L);
    if (__all_sync(0xffffffffu, is_finite(sum))) return sum.value();
    return lanes_sum2(a.value(), b.value(), L);
}

// Sum of one double per lane over a warp, valid in lane 0 (fixed order).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    return v;
}

}  // namespace mtdao
