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

// the error of t = a + b (Knuth's two-sum)
__device__ __forceinline__ float two_sum_error(float a, float b, float t) {
    const float bp = t - a;
    return (a - (t - bp)) + (b - bp);
}

// value and error term of a sum of floats
struct PairSum {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        e += two_sum_error(s, x, t);
        s = t;
    }
};

// the same for sums of many: every few terms fold() adds the error term of those
// to the others', with an error term of its own (a plain error term of hundreds of
// cells rounds, often always the same way, by 2^-50 of the sum)
struct LongSum : PairSum {
    float far = 0.f, rest = 0.f;
    __device__ __forceinline__ void fold() {
        const float t = far + e;
        rest += two_sum_error(far, e, t);
        far = t;
        e = 0.f;
    }
    __device__ __forceinline__ float error() const { return (e + rest) + far; }
};

// A sum of products with the products' own errors.  Those are kept apart from
// the sum's: the latter are few bits and mostly add up exactly, in one term they
// would make each other round.
struct ProductSum : LongSum {
    float q = 0.f;
    __device__ __forceinline__ void add_product(float a, float b) {
        const float p = __fmul_rn(a, b);  // (never part of an FMA: the sum is of the rounded product)
        add(p);
        q += fmaf(a, b, -p);
    }
    __device__ __forceinline__ float error() const { return LongSum::error() + q; }
};

// A sum of squares: the errors of squares are not even in sign, so that their sum
// grows with the number of cells and rounds always the same way; it gets an error
// term of its own.
struct SquareSum : LongSum {
    PairSum q;
    __device__ __forceinline__ void add_square(float a) {
        const float p = __fmul_rn(a, a);
        add(p);
        q.add(fmaf(a, a, -p));
    }
    __device__ __forceinline__ float product_error() const { return q.e + q.s; }
};

// the same for every number on the integer pipe, where subnormal ones are common
// (sums over the empty tails of a distribution)
__device__ __forceinline__ double widen_any(float x) {
    const bool small = fabsf(x) < 0x1p-126f;
    const unsigned b = __float_as_uint(small ? x * 0x1p64f : x), m = b & 0x7fffffffu;
    const unsigned bias = small ? 0x34000000u : (m < 0x7f800000u ? 0x38000000u : 0x70000000u);
    return __hiloint2double((int)((b & 0x80000000u) | (m ? (m >> 3) + bias : 0u)), (int)(b << 29));
}

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
