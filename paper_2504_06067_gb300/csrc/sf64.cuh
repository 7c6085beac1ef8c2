// sf64.cuh -- correctly rounded FP64 division and square root of normal
// numbers on the integer pipes.
//
// GB300 issues one FP64 instruction of a warp every 18 cycles per SM with 60
// cycles of latency, so a division (137 cycles of the pipe, 565 of latency)
// or a square root (144, 590) of a warp costs more than some kernels' whole
// FP32 work, and the chains of dependent divisions in the intercept solve
// set the time of small generations.  Integer multiply-adds run at the full
// rate.  Method: a 24-bit FP32 estimate, Newton steps in 64-bit fixed point,
// then the exact remainder decides the last bit, as in any digit-recurrence
// proof: t = floor of the 54-bit result is right if its remainder is in
// range, whatever the error of the estimate (the estimate is within a few
// units of 2^-62, so t is off by at most one, which the remainder corrects).
// Round to nearest, ties to even, from the 54th bit and the remainder: the
// same value as __ddiv_rn / __dsqrt_rn.  Subnormal, zero, infinite and NaN
// operands and results near the exponent range take those functions.
// (Latencies and rates measured with chains of dependent operations in one
// and in sixteen warps of an SM.)
#pragma once
#include <cstdint>

#ifdef __CUDA_ARCH__
#define SF_HD __device__ __forceinline__
#else
#include <cmath>
#include <cstring>
#define SF_HD inline
#endif

namespace sf64 {

typedef unsigned long long u64;
typedef long long i64;

#ifdef __CUDA_ARCH__
SF_HD u64 bits(double x) { return (u64)__double_as_longlong(x); }
SF_HD double value(u64 b) { return __longlong_as_double((i64)b); }
SF_HD u64 mulhi(u64 a, u64 b) { return __umul64hi(a, b); }
SF_HD float rcp32(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
SF_HD float rsq32(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
SF_HD uint32_t f2u(float x) { return __float2uint_rz(x); }  // saturates
SF_HD float u2f(uint32_t x) { return __uint2float_rz(x); }
SF_HD double hw_div(double a, double b) { return __ddiv_rn(a, b); }
SF_HD double hw_sqrt(double a) { return __dsqrt_rn(a); }
#else
// host forms for the test of the arithmetic; sf_ulp shifts the FP32 estimates
extern int sf_ulp;
SF_HD u64 bits(double x)
{
    u64 b;
    memcpy(&b, &x, 8);
    return b;
}
SF_HD double value(u64 b)
{
    double x;
    memcpy(&x, &b, 8);
    return x;
}
SF_HD u64 mulhi(u64 a, u64 b) { return (u64)(((unsigned __int128)a * b) >> 64); }
SF_HD float shifted(float r)
{
    int i;
    memcpy(&i, &r, 4);
    i += sf_ulp;
    memcpy(&r, &i, 4);
    return r;
}
SF_HD float rcp32(float x) { return shifted(1.0f / x); }
SF_HD float rsq32(float x) { return shifted(1.0f / sqrtf(x)); }
SF_HD uint32_t f2u(float x) { return x >= 4294967296.0f ? 0xffffffffu : (uint32_t)x; }
SF_HD float u2f(uint32_t x) { return (float)x; }  // x < 2^24: exact
SF_HD double hw_div(double a, double b) { return a / b; }
SF_HD double hw_sqrt(double a) { return sqrt(a); }
#endif

// A divisor ready for divisions: mantissa (53 bits), exponent field and
// R = 2^126 / (m << 11) within a few units (1/b' for b' = m / 2^53 in
// [1/2, 1), scaled by 2^62).  exp 0: not a normal number.
struct Divisor {
    u64 m, R, b;
    int exp;
};

SF_HD Divisor divisor(double x)
{
    Divisor d;
    d.b = bits(x);
    const int e = (int)(d.b >> 52) & 2047;
    d.exp = e == 2047 ? 0 : e;
    d.m = (d.b & 0xfffffffffffffull) | (1ull << 52);
    const u64 B = d.m << 11;
    const uint32_t R0 = f2u(rcp32(u2f((uint32_t)(B >> 40))) * 18014398509481984.0f);  // 2^54: 1/b' x 2^30
    // e = 1 - b' r0 (below 2^-21), r1 = r0 + r0 e
    const i64 e1 = (i64)((1ull << 62) - mulhi(B, (u64)R0 << 32));
    const u64 R1 = ((u64)R0 << 32) + (u64)(((i64)R0 * (e1 >> 13)) >> 17);
    // and once more (e below 2^-40)
    const i64 e2 = (i64)((1ull << 62) - mulhi(B, R1));
    d.R = R1 + (u64)(((i64)(R1 >> 32) * e2) >> 30);
    return d;
}

// RN(a / d)
SF_HD double div(double a, const Divisor& d)
{
    const u64 ab = bits(a);
    const int ea = (int)(ab >> 52) & 2047;
    const int er = ea - d.exp + 1023;
    if (ea == 0 || ea == 2047 || d.exp == 0 || er < 2 || er > 2045) {
        if ((ab << 1) == 0ull && d.exp != 0) return value((ab ^ d.b) & (1ull << 63));  // a zero, as common as any value
        return hw_div(a, value(d.b));
    }
    const u64 ma = (ab & 0xfffffffffffffull) | (1ull << 52);
    const int lt = ma < d.m ? 1 : 0;  // quotient below 1: one more bit
    const u64 q = mulhi(ma << 11, d.R);  // quotient x 2^62
    u64 t = q >> (9 - lt);               // 54 bits
    i64 rem = (i64)((ma << (53 + lt)) - t * d.m);  // modulo 2^64; the true value is small
    if (rem < 0) {
        --t;
        rem += (i64)d.m;
    } else if (rem >= (i64)d.m) {
        ++t;
        rem -= (i64)d.m;
    }
    u64 mant = t >> 1;
    mant += (t & 1ull) & ((rem != 0 ? 1ull : 0ull) | (mant & 1ull));
    return value((((u64)(er - lt - 1)) << 52) + mant | ((ab ^ d.b) & (1ull << 63)));
}

SF_HD double div(double a, double b) { return div(a, divisor(b)); }

// comparisons of the FP64 pipe (110 cycles of latency each) as integer tests
SF_HD bool is_zero(double x) { return (bits(x) << 1) == 0ull; }
SF_HD bool is_negative(double x) { return (i64)bits(x) < 0; }  // (-0.0 too)

// RN(sqrt(x))
SF_HD double sqrt_rn(double x)
{
    const u64 xb = bits(x);
    const int e = (int)(xb >> 52);  // the sign bit makes it larger than 2047
    if (e == 0 || e >= 2047) return xb == 0ull ? x : hw_sqrt(x);
    const u64 m = (xb & 0xfffffffffffffull) | (1ull << 52);
    const int odd = (e & 1) ^ 1;             // exponent e - 1023 odd
    const u64 A = m << (10 + odd);           // A in [1, 4) x 2^62
    const uint32_t Y0 = f2u(rsq32(u2f((uint32_t)(A >> 40))) * 8796093022208.0f);  // 2^43: y in (1/2, 1] x 2^32
    const i64 e1 = (i64)((1ull << 62) - mulhi(A, (u64)Y0 * Y0));  // 1 - A y^2
    const u64 Y1 = ((u64)Y0 << 31) + (u64)(((i64)Y0 * (e1 >> 13)) >> 19);  // x 2^63
    const u64 S1 = mulhi(A, Y1) << 2;                              // s = A y x 2^63
    const i64 r = (i64)(A - mulhi(S1, S1));                        // A - s^2
    const u64 S = S1 + (u64)(((i64)(Y1 >> 32) * r) >> 31);
    u64 t = S >> 10;  // 54 bits
    i64 rem = (i64)((m << (54 + odd)) - t * t);
    if (rem < 0) {
        --t;
    } else if (rem > (i64)(2 * t)) {
        ++t;
    }
    const u64 mant = (t >> 1) + (t & 1ull);  // a square root is never halfway
    const int h = (e - 1023 - odd) >> 1;     // e - 1023 - odd is even
    return value(((u64)(h + 1022) << 52) + mant);
}

}  // namespace sf64
