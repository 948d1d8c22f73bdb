// float_sum.cuh - sums of FP32 numbers that lose no more than FP64 sums would.
#pragma once

#ifndef __CUDACC__  // (plain C++: the arithmetic is checked on the host)
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace mdgb {

// Additions that are never fused with a product before them (a term may be one: with its product unrounded
// in the sum and rounded in the error, the error is wrong).
__host__ __device__ __forceinline__ float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}
__host__ __device__ __forceinline__ float sub_rn(float a, float b) { return add_rn(a, -b); }

// s + e = a + b exactly, s = a + b rounded (Knuth's two-sum); e does not depend on the order of a and b.
__host__ __device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = add_rn(a, b);
    const float t = sub_rn(s, a);
    e = add_rn(sub_rn(a, sub_rn(s, t)), sub_rn(b, t));
}

// The sum of FP32 numbers in three floats: the rounding error of every addition to hi goes to mid, that
// of every addition to mid to lo, and only the additions to lo round (at 2^-72 of the largest partial
// sum, where an FP64 sum rounds at 2^-53).  FP64 additions and conversions would hold a warp as
// long as some 60 FP32 operations each.  A term that is not finite, or a partial sum beyond FP32's range,
// leaves get() not finite: the caller then adds the terms again in FP64.
struct FloatSum {
    float hi = 0.f, mid = 0.f, lo = 0.f;

    __host__ __device__ __forceinline__ void add(float x) {
        float e1, e2;
        two_sum(hi, x, hi, e1);
        two_sum(mid, e1, mid, e2);
        lo = add_rn(lo, e2);
    }

    // The other of two sums; the same bits whichever of the two takes it.
    __host__ __device__ __forceinline__ void add(const FloatSum& o) {
        float e1, e2, e3, m;
        two_sum(hi, o.hi, hi, e1);
        two_sum(mid, o.mid, m, e2);
        two_sum(m, e1, mid, e3);
        lo = add_rn(add_rn(lo, o.lo), add_rn(e2, e3));
    }

    __host__ __device__ __forceinline__ double get() const { return (double)hi + ((double)mid + (double)lo); }
};

#ifdef __CUDACC__
__device__ __forceinline__ FloatSum lane_xor(const FloatSum& s, int o) {
    return FloatSum{__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.mid, o),
                    __shfl_xor_sync(0xffffffffu, s.lo, o)};
}
#endif

}  // namespace mdgb
