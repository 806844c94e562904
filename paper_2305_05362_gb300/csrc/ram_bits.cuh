// FP64 arithmetic with few FP64 instructions: the FP64 pipe takes a warp instruction
// every 16 cycles of an SM, the integer pipe 32 times as many.  Comparisons, signs,
// minima of magnitudes and scalings by powers of two work on the bits (a magnitude's
// order is its bits'), quotients are a cubic Newton step from the hardware's
// reciprocal approximation.  Subnormal magnitudes count as zero in the scalings;
// callers keep values of 2^1000 or more, infinities and NaN away from these forms.
#pragma once

#include <cuda_runtime.h>

namespace ram {

__device__ __forceinline__ unsigned long long mag(double x)
{
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
// magnitude times 2^k, k = 1 or 2 (subnormals: 0)
__device__ __forceinline__ unsigned long long mag_up(unsigned long long m, int k)
{
    return (m >> 52) == 0 ? 0ull : m + ((unsigned long long)k << 52);
}
// |x| > |y|, false where x is NaN
__device__ __forceinline__ bool mag_above(double x, double y)
{
    return mag(x) > mag(y) && mag(x) <= 0x7ff0000000000000ull;
}
__device__ __forceinline__ unsigned long long mag_min(unsigned long long a, unsigned long long b)
{
    return a < b ? a : b;
}
// the magnitude m with s's sign, zero where s and t differ in sign
__device__ __forceinline__ double mag_signed(unsigned long long m, double s, double t)
{
    const int hs = __double2hiint(s), ht = __double2hiint(t);
    const unsigned long long v = m | ((unsigned long long)(hs & 0x80000000) << 32);
    return (hs ^ ht) < 0 ? 0.0 : __longlong_as_double((long long)v);
}
__device__ __forceinline__ double half_of(double x)
{
    const long long b = __double_as_longlong(x);
    return ((b >> 52) & 0x7ff) < 2 ? 0.0 : __longlong_as_double(b - (1ll << 52));
}
// half the van Leer slope, dl dr / (dl + dr) where dl and dr have one sign, else 0
__device__ __forceinline__ double half_vl_bits(double dl, double dr)
{
    const double p = dl * dr, s = dl + dr;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(s));
    const double e = fma(-s, r, 1.0);
    const double u = p * r;
    const double h = fma(u, fma(e, e, e), u);
    const bool one_sign = (__double2hiint(dl) ^ __double2hiint(dr)) >= 0;
    // s normal: both zero, or sums too small for the reciprocal, have no slope
    return one_sign && (mag(s) >> 52) > 1 ? h : 0.0;
}
// the high word of a magnitude (ordered as the magnitudes are), and its bounds above
__device__ __forceinline__ unsigned mag_hi(double x)
{
    return (unsigned)__double2hiint(x) & 0x7fffffffu;
}
constexpr unsigned kMagBig = 0x7e700000u;    // 2^1000; infinity and NaN above
constexpr unsigned kMagSmall = 0x26f00000u;  // 2^-400

// x 2^k for a normal x with a normal result
__device__ __forceinline__ double scale_pow2(double x, int k)
{
    return __hiloint2double(__double2hiint(x) + (k << 20), __double2loint(x));
}

// d rounded to double (halves away from zero), on the integer pipe
__device__ __forceinline__ double u64_to_double(unsigned long long d)
{
    const int lz = __clzll((long long)d);
    const unsigned long long m = d << (lz & 63);  // the leading one at bit 63
    const unsigned long long v = ((unsigned long long)(1023 + 63 - 1 - lz) << 52) + (m >> 11) +
                                 ((m >> 10) & 1ull);
    return d == 0 ? 0.0 : __longlong_as_double((long long)v);
}

// 1 / x for a normal x whose reciprocal is normal: from r0 with e = 1 - x r0, r0 (1 + e
// + e^2) leaves e^3, below rounding (within 1 ulp)
__device__ __forceinline__ double rcp_newton(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

}  // namespace ram
