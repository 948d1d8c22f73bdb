// fp64_math.cuh - FP64 reciprocals in few FP64 operations, shared by the FP64 kernels.
#pragma once

#include "fixpt.cuh"

namespace mdgb {

// 1/x to within about an ulp: the hardware's approximate reciprocal, refined by two
// Newton-Raphson steps y <- y + y (1 - x y), each of which doubles the correct bits (a
// seed good to 2^-14 or better reaches full precision).  For x = 0 the result is not
// finite, and the force kernels flag the non-finite force.
__device__ __forceinline__ double rcp_nr(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double e = fma(-x, y, 1.0);
        y = fma(y, e, y);
    }
    return y;
}

// The FP32 number of a double's upper half (20 mantissa bits, truncated; 0 below FP32's range).
__device__ __forceinline__ float upper_f32(double x) {
    const int h = __double2hiint(x);
    const int t = max((h & 0x7fffffff) - (896 << 20), 0);
    return __int_as_float((h & (int)0x80000000) | (t << 3));
}

// 1/x to within about an ulp in three FP64 operations, for x well inside FP32's range
// (2^-100 .. 2^126): from an FP32 seed y (error e = 1 - x y of 2^-22) one step y (1 + e + e^2) of
// Householder's third-order iteration leaves e^3.  Other x, zero among them, take rcp_nr.
static __device__ __noinline__ double rcp_nr_far(double x) { return rcp_nr(x); }  // (a call: not computed for every x)

__device__ __forceinline__ double rcp_cubic(double x) {
    const unsigned h = (unsigned)__double2hiint(x) - (896u << 20);  // exponent as FP32 has it
    if (h - (27u << 20) >= (226u << 20)) return rcp_nr_far(x);
    const float xf = __int_as_float((int)__funnelshift_l((unsigned)__double2loint(x), h, 3));
    const int yf = __float_as_int(rcp_approx(xf));
    const double y = __hiloint2double((yf >> 3) + (896 << 20), yf << 29);
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

}  // namespace mdgb
