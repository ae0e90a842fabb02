// FP64 arithmetic for a GPU whose FP64 pipe is narrow.  GB300 issues a
// double-precision instruction of a warp in 16 cycles per SM against a
// quarter of a cycle in FP32, so the FP64 kernels are bound by the number of
// FP64 instructions alone.  Comparisons are done on the bit patterns (integer
// pipe), and reciprocals and reciprocal square roots start from the special
// function unit's 20-bit approximations, refined by one third-order step of
// Householder's method on the defining equation: three FP64 instructions for
// a reciprocal and five for a reciprocal square root instead of a division or
// square root rounded correctly.  The figures at the functions are the largest
// errors over 4 million random operands of exponents -300 to 300, in units of the
// result's last place.  The seeds take normal operands and give normal results:
// of a zero, subnormal or infinite operand, or one whose reciprocal is subnormal,
// rcp64 makes NaN or 0, and rsqrt64 infinity, 0 or NaN.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace hyd {

__device__ __forceinline__ long long dbits(double v) { return __double_as_longlong(v); }
__device__ __forceinline__ unsigned dhi(double v) { return (unsigned)__double2hiint(v); }

// 0 < v (v not NaN), without the FP64 pipe
__device__ __forceinline__ bool dpos(double v) {
    return (unsigned long long)dbits(v) - 1ull < 0x7ff0000000000000ull;
}

// v positive, normal and finite
__device__ __forceinline__ bool dnormal(double v) {
    return dhi(v) - 0x00100000u < 0x7fe00000u;
}

// v zero (of either sign)
__device__ __forceinline__ bool dzero(double v) {
    return ((dhi(v) << 1) | (unsigned)__double2loint(v)) == 0u;
}

// 0 <= v for a result of arithmetic (whose NaN is 0x7fffffff ffffffff), from the high
// word: -0 counts, as do negative numbers above -2^-1042
__device__ __forceinline__ bool dge0(double v) {
    return dhi(v) <= 0x7ff00000u || dhi(v) == 0x80000000u;
}

// v < 0 (neither -0 nor NaN)
__device__ __forceinline__ bool dneg(double v) {
    const unsigned long long b = (unsigned long long)dbits(v);
    return b > 0x8000000000000000ull && b <= 0xfff0000000000000ull;
}

// integer with the order of the doubles (-0 just below +0; NaN beyond infinity)
__device__ __forceinline__ long long dkey(double v) {
    const long long b = dbits(v);
    return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
}
__device__ __forceinline__ double dunkey(long long k) {
    return __longlong_as_double(k ^ (long long)((unsigned long long)(k >> 63) >> 1));
}
__device__ __forceinline__ bool dlt(double a, double b) { return dkey(a) < dkey(b); }
// a < b for a, b >= 0 (false when a is NaN; b must not be: its bits are above all)
__device__ __forceinline__ bool dlt_pos(double a, double b) {
    return (unsigned long long)dbits(a) < (unsigned long long)dbits(b);
}
__device__ __forceinline__ double dmin_(double a, double b) { return dlt(b, a) ? b : a; }
__device__ __forceinline__ double dmax_(double a, double b) { return dlt(a, b) ? b : a; }
__device__ __forceinline__ double dabs_(double v) {
    return __longlong_as_double(dbits(v) & 0x7fffffffffffffffll);
}

__device__ __forceinline__ double rcp_seed(double x) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}

// 1 / x (0.51 units): with e = 1 - x r, 1 / x = r / (1 - e) = r (1 + e + e^2) + O(e^3)
__device__ __forceinline__ double rcp64(double x) {
    const double r = rcp_seed(x);
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}

// 1 / x to 2^-39.9 (one Newton step): for factors of small corrections
__device__ __forceinline__ double rcp40(double x) {
    const double r = rcp_seed(x);
    return fma(r, fma(-x, r, 1.0), r);
}

// 1 / sqrt(x) (1.0 units), x positive, normal and finite (dnormal first where
// anything else can occur): with e = 1 - x r^2, (1 - e)^(-1/2) = 1 + e/2 + 3 e^2/8 + O(e^3)
__device__ __forceinline__ double rsqrt64(double x) {
    const double r = rsqrt_seed(x);
    const double e = fma(-x * r, r, 1.0);
    return fma(r, e * fma(0.375, e, 0.5), r);
}

// sqrt(x) of what rsqrt64 does not take: 0 of zeros and positive subnormals,
// infinity of itself, NaN of negative numbers and NaN
__device__ __forceinline__ double sqrt_rest(double x) {
    const unsigned long long b = (unsigned long long)dbits(x);
    if (b < 0x0010000000000000ull || (b << 1) == 0ull) return 0.0;
    return __longlong_as_double(b == 0x7ff0000000000000ull ? 0x7ff0000000000000ll
                                                           : 0x7ff8000000000000ll);
}

// sqrt(x) (0.50 units): the residual x - s^2, exact in a fused multiply-add,
// corrects s (Markstein, IBM J. Res. Dev. 34, 1990)
__device__ __forceinline__ double sqrt64(double x) {
    const double r = rsqrt64(x);
    const double s = x * r;
    const double t = fma(fma(-s, s, x), 0.5 * r, s);
    // (a negative operand's seed is NaN)
    if (((dhi(x) >> 20) & 0x7ffu) - 1u >= 0x7feu) return sqrt_rest(x);
    return t;
}

// a / b from y = 1/b (within an ulp): each step adds the exactly computed
// remainder a - b q times y (Markstein, 1990).  One step leaves the quotient within
// a hair of half an ulp (0.50 units, none of 4 million rounded wrongly); two give
// the correctly rounded one (the remainder of a quotient within one ulp is exact,
// and its product with y is far below the distance of any quotient from a rounding
// boundary).
__device__ __forceinline__ double div1(double a, double b, double y) {
    const double q = a * y;
    return fma(fma(-q, b, a), y, q);
}
__device__ __forceinline__ double div2(double a, double b, double y) {
    const double q = div1(a, b, y);
    return fma(fma(-q, b, a), y, q);
}

// finite, without the FP64 pipe
__device__ __forceinline__ bool dfinite(double v) {
    return ((unsigned)(dbits(v) >> 52) & 0x7ffu) != 0x7ffu;
}

// floor(q 2^64) for 0 <= q < 1 (0 below 2^-64)
__device__ __forceinline__ unsigned long long fixed64(double q) {
    const unsigned long long b = (unsigned long long)dbits(q);
    const int e = (int)(b >> 52);
    const unsigned long long m = (b & 0xfffffffffffffull) | (1ull << 52);
    const int shift = e - 1011;
    return shift >= 0 ? m << shift : shift > -64 && e > 0 ? m >> -shift : 0ull;
}

// t^n, n >= 1 uniform over the warp
__device__ __forceinline__ double ipow64(double t, int n) {
    double r = (n & 1) ? t : 1.0;
    for (n >>= 1; n > 0; n >>= 1) {
        t *= t;
        if (n & 1) r *= t;
    }
    return r;
}

}  // namespace hyd
