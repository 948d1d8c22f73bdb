// float_sum.cuh - sums of FP32 numbers that lose no more than FP64 sums would.
#pragma once

#ifdef __CUDACC__
#include "fixpt.cuh"
#else  // (plain C++: the arithmetic is checked on the host)
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace mdgb {

// s + e = a + b exactly, s = a + b rounded (Knuth's two-sum); e does not depend on the order of a and b.
// No argument may be a product that the compiler could fuse into the additions (the error would then be
// that of the rounded product): products go to FloatSum2 below, whose additions are not fused.
__host__ __device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float t = s - a;
    e = (a - (s - t)) + (b - t);
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
        lo += e2;
    }

    // The other of two sums; the same bits whichever of the two takes it.
    __host__ __device__ __forceinline__ void add(const FloatSum& o) {
        float e1, e2, e3, m;
        two_sum(hi, o.hi, hi, e1);
        two_sum(mid, o.mid, m, e2);
        two_sum(m, e1, mid, e3);
        lo = (lo + o.lo) + (e2 + e3);
    }

    __host__ __device__ __forceinline__ double get() const { return (double)hi + ((double)mid + (double)lo); }
};

#ifdef __CUDACC__
__device__ __forceinline__ FloatSum lane_xor(const FloatSum& s, int o) {
    return FloatSum{__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.mid, o),
                    __shfl_xor_sync(0xffffffffu, s.lo, o)};
}

// Two such sums in packed FP32x2 registers: the same operations in half the instructions, none of them fused
// with a product before it.  (The reduction of the energies runs the scalar form: its additions are plain
// ones that leave the compiler its order of loads, 17.9 us at 1,048,576 atoms against 27.6.)
__device__ __forceinline__ void two_sum2(f2_t a, f2_t b, f2_t& s, f2_t& e) {
    s = f2_add(a, b);
    const f2_t t = f2_sub(s, a);
    e = f2_add(f2_sub(a, f2_sub(s, t)), f2_sub(b, t));
}

struct FloatSum2 {
    f2_t hi = 0ull, mid = 0ull, lo = 0ull;

    __device__ __forceinline__ void add(float x, float y) {
        f2_t e1, e2;
        two_sum2(hi, f2_pack(x, y), hi, e1);
        two_sum2(mid, e1, mid, e2);
        lo = f2_add(lo, e2);
    }
    __device__ __forceinline__ void add(const FloatSum2& o) {
        f2_t e1, e2, e3, m;
        two_sum2(hi, o.hi, hi, e1);
        two_sum2(mid, o.mid, m, e2);
        two_sum2(m, e1, mid, e3);
        lo = f2_add(f2_add(lo, o.lo), f2_add(e2, e3));
    }
    __device__ __forceinline__ FloatSum half(bool second) const {
        float h[2], m[2], l[2];
        f2_unpack(hi, h[0], h[1]);
        f2_unpack(mid, m[0], m[1]);
        f2_unpack(lo, l[0], l[1]);
        return second ? FloatSum{h[1], m[1], l[1]} : FloatSum{h[0], m[0], l[0]};
    }
};

__device__ __forceinline__ FloatSum2 lane_xor(const FloatSum2& s, int o) {
    return FloatSum2{__shfl_xor_sync(0xffffffffu, s.hi, o), __shfl_xor_sync(0xffffffffu, s.mid, o),
                     __shfl_xor_sync(0xffffffffu, s.lo, o)};
}

// The same interface over FP64 sums.
struct DoubleSum {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void add(const DoubleSum& o) { v += o.v; }
    __device__ __forceinline__ double get() const { return v; }
};

__device__ __forceinline__ DoubleSum lane_xor(const DoubleSum& s, int o) {
    return DoubleSum{__shfl_xor_sync(0xffffffffu, s.v, o)};
}

struct DoubleSum2 {
    double a = 0.0, b = 0.0;
    __device__ __forceinline__ void add(double x, double y) {
        a += x;
        b += y;
    }
    __device__ __forceinline__ void add(const DoubleSum2& o) { add(o.a, o.b); }
    __device__ __forceinline__ DoubleSum half(bool second) const { return DoubleSum{second ? b : a}; }
};

__device__ __forceinline__ DoubleSum2 lane_xor(const DoubleSum2& s, int o) {
    return DoubleSum2{__shfl_xor_sync(0xffffffffu, s.a, o), __shfl_xor_sync(0xffffffffu, s.b, o)};
}
#endif

}  // namespace mdgb
