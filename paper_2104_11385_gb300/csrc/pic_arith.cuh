// pic_arith.cuh -- the arithmetic of the Boris push: double, and float with
// conversions by integer work on the IEEE-754 bits (on GB300 every FP64
// instruction, conversions included, issues at 1/64 of the FP32 rate).
#pragma once
#include <cuda_runtime.h>

// ---- plain FP32 (the FP32 variant): conversions by integer work as well
static __device__ __noinline__ float f32_from_slow(double x) { return __double2float_rn(x); }
static __device__ __noinline__ double f64_from_slow(float f) { return (double)f; }

// double -> float, rounded to 24 bits (ties away from zero on the magnitude)
// on the bit pattern; zero, and magnitudes outside [2^-100, 2^127), take the
// conversion instruction out of line
__device__ __forceinline__ float f32_from(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned long long u = b & 0x7FFFFFFFFFFFFFFFull;
    const int be = (int)(u >> 52);
    const unsigned sgn = (unsigned)(b >> 32) & 0x80000000u;
    if (be >= 1023 - 100 && be <= 1023 + 126)
        return __uint_as_float(sgn | (unsigned)(((u + (1ull << 28)) >> 29) - (896ull << 23)));
    if (u == 0ull) return __uint_as_float(sgn);
    return f32_from_slow(x);
}

// float -> double, exact: exponent rebias and mantissa << 29 for normal floats
__device__ __forceinline__ double f64_from(float f) {
    const unsigned b = __float_as_uint(f), a = b & 0x7FFFFFFFu;
    const unsigned long long sg = (unsigned long long)(b & 0x80000000u) << 32;
    if (a >= 0x00800000u && a < 0x7F800000u)
        return __longlong_as_double((long long)(sg | (((unsigned long long)a + (896ull << 23)) << 29)));
    if (a == 0u) return __longlong_as_double((long long)sg);
    return f64_from_slow(f);
}

// ---- one arithmetic interface for double and float
template <class R>
struct Arith;

template <>
struct Arith<double> {
    __device__ static __forceinline__ double from(double x) { return x; }
    __device__ static __forceinline__ double to(double x) { return x; }
    // 1/sqrt(x) for x >= 1 (1 + |u|^2): the hardware estimate y (about 20 bits)
    // and one step of Householder's method of order 2 (A. S. Householder, The
    // Numerical Treatment of a Single Nonlinear Equation, 1970) for y^-2 - x, that
    // is the first terms of the binomial series: with e = 1 - x y^2,
    // 1/sqrt(x) = y (1 - e)^(-1/2) = y + y e (1/2 + 3/8 e) + O(e^3); five FP64
    // instructions against seven for two Newton-Raphson steps.  Within
    // 1.24 x 2^-53 of the exact value, 0.48 rms (two Newton-Raphson steps: 1.23, 0.48)
    __device__ static __forceinline__ double rsqrt(double x) {
        double y;
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        const double e = ::fma(-x * y, y, 1.0);
        return ::fma(y * e, ::fma(0.375, e, 0.5), y);
    }
    // 2/x for x >= 1: the hardware reciprocal estimate y (about 20 bits), doubled
    // through its exponent, and one step of the same method for 1/y - x, the
    // geometric series: with e = 1 - x y, 1/x = y (1 + e + e^2) + O(e^3).  Within
    // 1.00 x 2^-53 of the exact value, 0.44 rms (two Newton-Raphson steps: the same)
    __device__ static __forceinline__ double two_over(double x) {
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        const double e = ::fma(-x, y, 1.0);
        const double y2 = __hiloint2double(__double2hiint(y) + 0x100000, __double2loint(y));
        return ::fma(y2, ::fma(e, e, e), y2);
    }
    // x + v dt/dx
    __device__ static __forceinline__ double move(double v, double k, double x) { return ::fma(v, k, x); }
    __device__ static __forceinline__ double c(double x) { return x; }
};

template <>
struct Arith<float> {
    __device__ static __forceinline__ float from(double x) { return f32_from(x); }
    __device__ static __forceinline__ double to(float x) { return f64_from(x); }
    __device__ static __forceinline__ float rsqrt(float x) { return rsqrtf(x); }
    __device__ static __forceinline__ float two_over(float x) { return 2.0f * __frcp_rn(x); }
    __device__ static __forceinline__ float c(double x) { return static_cast<float>(x); }
};
