// vp_sum.cuh -- sums of floats in more than float precision without the FP64
// pipe (two FMA lanes per SM and clock, conversions included).
#pragma once

#include <cuda_runtime.h>

namespace vp_sum {

// (double)x on the bits of a normal number or zero; other numbers take the
// conversion, out of line (as a predicated instruction it occupies the FP64 pipe
// for every number)
__device__ __noinline__ inline double widen_rare(float x) { return (double)x; }
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    const unsigned hi = (b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u);
    double d = __hiloint2double((int)hi, (int)(b << 29));
    if (m != 0u && m - 0x00800000u >= 0x7f000000u) d = widen_rare(x);
    return d;
}

// value and error term of a sum of floats (Knuth's two-sum)
struct PairSum {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        const float bp = t - s;
        e += (s - (t - bp)) + (x - bp);
        s = t;
    }
    // a b, both rounding errors kept
    __device__ __forceinline__ void add_product(float a, float b) {
        const float p = a * b;
        add(p);
        e += fmaf(a, b, -p);
    }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace vp_sum
