// real64.cuh -- FP64 building blocks of the kernels that the FP64 pipe bounds.
//
// GB300 issues 2 FP64 lanes per SM and clock, 1/64 of its FP32 rate, and a
// comparison, minimum, conversion or rounding of doubles takes the same slot
// as a multiply-add.  These functions keep to the fewest FP64 operations and
// leave the rest (signs, range checks, integer parts) to the integer units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gcb {

// 0, denormal, negative, infinite or NaN (not a positive normal number)
__device__ __forceinline__ bool not_pos_normal(double x)
{
    return (unsigned)__double2hiint(x) - 0x00100000u >= 0x7fe00000u;
}
__device__ __forceinline__ bool finite64(double x)
{
    return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;
}
// a > b for a, b >= 0 (a NaN counts as larger than every number)
__device__ __forceinline__ bool gt_nonneg(double a, double b)
{
    return __double_as_longlong(a) > __double_as_longlong(b);
}

// 1/x and 1/sqrt(x): the hardware's approximation (PTX rcp.approx.ftz.f64 and
// rsqrt.approx.ftz.f64, about 20 bits) and one step of Householder's
// third-order iteration (A. S. Householder, The Numerical Treatment of a
// Single Nonlinear Equation, 1970): with the residual e = 1 - x y (1 - x y^2)
// the step y (1 + e + e^2) (y (1 + e/2 + 3 e^2/8)) leaves a relative error of
// order e^3.  Within 1 ulp of the exact value for normal results; 3 and 5 FP64
// operations, where the IEEE quotient and 1.0 / sqrt(x) take about 10 and 20.
// Infinite and zero arguments give their limits, NaN and negative arguments
// of the root NaN; denormals count as 0, denormal results are flushed.
__device__ __forceinline__ double rcp64(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    const double q = fma(e, e, e);
    const double r = fma(y, q, y);
    return not_pos_normal(fabs(y)) || !finite64(x) ? y : r;
}
__device__ __forceinline__ double rsqrt64(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = x * y;
    const double e = fma(-h, y, 1.0);
    const double p = fma(e, 0.375, 0.5);
    const double r = fma(e * y, p, y);
    return not_pos_normal(x) ? y : r;
}
// sqrt(x) = x / sqrt(x): within 2 ulp; 0 and infinity map to themselves
__device__ __forceinline__ double sqrt64(double x)
{
    const double r = x * rsqrt64(x);
    return not_pos_normal(x) && __double2hiint(x) >= 0 ? x : r;
}

// A float as a double, by its bits: the conversion instruction takes an FP64
// pipe slot.  Denormals: flushed to zero (FTZ, as the conversion does in the
// units compiled with that flag), else converted by the instruction (the asm is
// volatile, so that it is not issued for every value and then selected).
template <bool FTZ>
__device__ __forceinline__ double widen(float f)
{
    const unsigned b = __float_as_uint(f), a = b & 0x7fffffffu;
    const bool norm = a >= 0x00800000u;
    // exponent bias 1023 - 127; infinities and NaN to the top exponent
    const unsigned h = (a >> 3) + (a >= 0x7f800000u ? 0x70000000u : 0x38000000u);
    double r = __hiloint2double((int)((b & 0x80000000u) | (norm ? h : 0u)),
                                (int)(norm ? b << 29 : 0u));
    if (!FTZ && a - 1u < 0x007fffffu) asm volatile("cvt.f64.f32 %0, %1;" : "=d"(r) : "f"(f));
    return r;
}
template <bool FTZ>
__device__ __forceinline__ double widen(double f) { return f; }

// floor(s): its value, and as an integer clamped to [-n, n].  Adding 1.5 2^52
// rounded down leaves the floor in the low bits of the sum (exact for
// |s| < 2^51; beyond, and for NaN, the integer clamps).  2 FP64 additions in
// place of a rounding, two comparisons and a conversion.
__device__ __forceinline__ double floor64(double s, int n, int &k)
{
    const double M = 6755399441055744.0;   // 1.5 2^52
    const double t = __dadd_rd(s, M);
    const long long d = __double_as_longlong(t) - 0x4338000000000000LL;
    k = d > n ? n : (d < -(long long)n ? -n : (int)d);
    return t - M;
}

// l i = k + t: k = floor(l i) clamped to [-n, n] and t in [0, 1] (1 only where
// a product just below an integer rounds to it), from the product as it is,
// not rounded first.  3 FP64 operations where the product, floor64 and the
// difference take 4; every interpolation of an FP64 push has one an axis, and
// the push is bound by their number (8 steps of 2^20 particles, 2D, 15.24 ms
// before and 14.70 after; 3D, 3e5 particles, 6.07 and 5.92).
__device__ __forceinline__ double split64(double l, double i, int n, int &k)
{
    const double M = 6755399441055744.0;
    const double t = __fma_rd(l, i, M);
    const long long d = __double_as_longlong(t) - 0x4338000000000000LL;
    k = d > n ? n : (d < -(long long)n ? -n : (int)d);
    return fma(l, i, M - t);
}

}  // namespace gcb
