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
// them, so the pair stays good to about 2^-46 of the sum (fp64 costs 16 issue
// cycles an instruction on this chip, this some seven).
__device__ __forceinline__ Kahan operator+(const Kahan &a, const Kahan &b) {
    Kahan r;
    r.s = a.s + b.s;
    const float t = r.s - a.s;
    const float err = (a.s - (r.s - t)) + (b.s - t);   // a.s + b.s = r.s + err exactly
    r.c = (a.c + b.c) - err;
    return r;
}

// Sum over aligned groups of `lanes` lanes (a power of two up to 32), the same
// in every lane of the group.
__device__ __forceinline__ Kahan lanes_sum(Kahan v, int lanes) {
    for (int off = lanes >> 1; off > 0; off >>= 1) {
        Kahan o;
        o.s = __shfl_xor_sync(0xffffffffu, v.s, off);
        o.c = __shfl_xor_sync(0xffffffffu, v.c, off);
        v = v + o;
    }
    return v;
}

// Sum of one double per lane over a warp, valid in lane 0 (fixed order).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    return v;
}

}  // namespace mtdao
