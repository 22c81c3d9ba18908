// wb_math.cuh -- reciprocals and square roots of the sweep kernels, and the
// arithmetic they share over a scalar (FP64) or a pair of FP32 lanes.
//
// FP64 division and square roots: the hardware's approximate reciprocal (root)
// has about 20 good bits; one step of the third-order iteration of
// Householder's family takes that to the rounding level:
//   1/x:       e = 1 - x y,    y' = y (1 + e + e^2)
//   1/sqrt(x): e = 1 - x y^2,  y' = y (1 + e/2 + 3 e^2/8)
// in 3 and 5 operations of the narrow FP64 pipe, which bounds the FP64 sweep.
// Arguments outside the normal range (zero, subnormal, infinite, negative,
// NaN, or a reciprocal that would be subnormal) take CUDA's functions.
// Largest error seen over the binades: 1/x 1 ulp, 1/sqrt 1 ulp, sqrt 1 ulp
// (tests/test_gpu_math.py).
#pragma once
#include <cuda_runtime.h>

namespace wb {

// ---- scalar reciprocals and roots ---------------------------------------------
__device__ __forceinline__ bool normal_range(double x, unsigned lo, unsigned hi) {
    const unsigned h = (unsigned)__double2hiint(x);      // negative: above every bound
    return h >= lo && h < hi;
}
// 1/x for x > 0 known to lie in [2^-1000, 2^1000]
__device__ __forceinline__ double recip_inrange(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double recip(double x) {
    return normal_range(x, 0x00100000u, 0x7fc00000u) ? recip_inrange(x) : 1.0 / x;
}
__device__ __forceinline__ double rsq_root(double x) {
    if (!normal_range(x, 0x00100000u, 0x7ff00000u)) return rsqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double t = x * y;
    const double e = fma(-t, y, 1.0);
    return fma(fma(0.375, e, 0.5), y * e, y);
}
// sqrt(x) = x / sqrt(x), the same step applied to t = x y: e holds the
// rounding error of t as well
__device__ __forceinline__ double sq_root(double x) {
    if (!normal_range(x, 0x00100000u, 0x7ff00000u)) return sqrt(x);
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double t = x * y;
    const double e = fma(-t, y, 1.0);
    return fma(fma(0.375, e, 0.5), t * e, t);
}
// FP32: the compiler's forms (the FP32 sweeps are built with fast division
// and square root)
__device__ __forceinline__ float recip(float x) { return 1.0f / x; }
__device__ __forceinline__ float rsq_root(float x) { return rsqrtf(x); }
__device__ __forceinline__ float sq_root(float x) { return sqrtf(x); }

// The FP64 value of an FP32 number, formed from its bits with integer
// operations (IEEE 754 binary32 -> binary64 is exact: sign kept, exponent
// rebiased by 1023 - 127, mantissa widened by 29 zero bits; subnormals
// normalised, zero, infinities and NaN mapped to their binary64 forms).  The
// conversion instruction would run on the FP64 pipe, which is narrow on this
// GPU; with this only the sums do.
__device__ __forceinline__ double widen(float x) {
    const unsigned int u = __float_as_uint(x);
    const unsigned long long sign = (unsigned long long)(u >> 31) << 63;
    const unsigned int e = (u >> 23) & 0xffu;
    unsigned int m = u & 0x7fffffu;
    unsigned long long bits;
    if (e == 0xffu) {                       // infinity or NaN
        bits = sign | (0x7ffull << 52) | ((unsigned long long)m << 29);
    } else if (e != 0u) {                   // normal
        bits = sign | ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)m << 29);
    } else if (m == 0u) {                   // signed zero
        bits = sign;
    } else {                                // subnormal: value m 2^-149
        const int sh = __clz(m) - 8;        // shifts that bring the top bit to bit 23
        m = (m << sh) & 0x7fffffu;
        bits = sign | ((unsigned long long)(897 - sh) << 52) | ((unsigned long long)m << 29);
    }
    return __longlong_as_double((long long)bits);
}

// ---- one FP64 value or two FP32 lanes -------------------------------------------
template <class V> struct Lanes;
template <> struct Lanes<double> { using S = double; };
template <> struct Lanes<float2> { using S = float; };

template <class V> __device__ __forceinline__ V splat(typename Lanes<V>::S v);
template <> __device__ __forceinline__ double splat<double>(double v) { return v; }
template <> __device__ __forceinline__ float2 splat<float2>(float v) { return make_float2(v, v); }

__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vfms(double a, double b, double c) { return fma(a, b, -c); }
__device__ __forceinline__ double vrcp(double a) { return recip(a); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 vfms(float2 a, float2 b, float2 c) {      // a b - c
    return make_float2(fmaf(a.x, b.x, -c.x), fmaf(a.y, b.y, -c.y));
}
__device__ __forceinline__ float2 vrcp(float2 a) { return make_float2(recip(a.x), recip(a.y)); }
__device__ __forceinline__ double vabs(double a) { return fabs(a); }
__device__ __forceinline__ float2 vabs(float2 a) { return make_float2(fabsf(a.x), fabsf(a.y)); }

}  // namespace wb
