// gf_squares.cuh -- a warp's sum of squares of short floats, to float64's accuracy at float32's rate.
#pragma once

#include <cuda_runtime.h>

// A lane's share: squares of values of at most 12 significant bits (exact in float32 while they stay in its
// range) summed as three floats -- a running sum, the errors of its additions, the errors of theirs, each
// exact but for the last one's own (below 2^-60 of the sum over 32 squares) -- and added to a float64 sum
// at least every 32 squares.  So the float64 sum rounds 3 times where one that takes every square rounds
// 32 times.  The float64 conversion and multiply-add of every value took most of the copies' time (GB300's
// float64 rate).
struct SquareSum {
    float hi = 0.f, mid = 0.f, lo = 0.f;
    double acc = 0.0;
    // a = fl(a + b), returns the rounding error (Knuth's TwoSum)
    static __device__ __forceinline__ float two_sum(float &a, float b) {
        const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
        const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
        a = s;
        return e;
    }
    __device__ __forceinline__ void add(float v) {
        const float e = two_sum(hi, __fmul_rn(v, v));
        lo = __fadd_rn(lo, two_sum(mid, e));
    }
    __device__ __forceinline__ void flush() {
        acc += hi;
        acc += mid;
        acc += lo;
        hi = mid = lo = 0.f;
    }
    __device__ __forceinline__ double warp_total() {
        flush();
        double a = acc;
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        return a;
    }
};
