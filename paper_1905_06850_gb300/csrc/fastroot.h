// fastroot.h -- 1 / sqrt(x) and 1 / x in FP64 from an FP32 seed (host and
// device; the host build serves the tests).
//
// An FP64 warp instruction takes 64 cycles on a GB300 SM sub-partition even
// when one lane works, so the scalar chain of a small solve counts FP64
// instructions: six here for the reciprocal square root, four for the
// reciprocal.  The seed y (24 bits, relative error below 2^-20) comes from the
// FP32 units; one step of Householder's method of third order (Householder,
// "The Numerical Treatment of a Single Nonlinear Equation", 1970, Sec. 4.4)
// follows: with the residual e = 1 - x y^2 (y^2 is exact in FP64, so e has one
// rounding), 1/sqrt(x) = y (1 - e)^{-1/2} = y + y e (1/2 + 3/8 e + 5/16 e^2) +
// O(e^4); with e = 1 - x y, 1/x = y / (1 - e) = y + y (e + e^2 + e^3) +
// O(e^4).  |e| < 2^-18: the terms left out are below 2^-72, and the result has
// the rounding of the last operation (0.5 ulp) plus a few 2^-18 of one.
// Positive normal numbers (the reciprocal: either sign) whose result is
// normal; everything else takes the plain operation.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "fxsum.h"

namespace plcg {

// FP32 seeds of 1/sqrt(m) and 1/m, m in [1, 4).
PLCG_HD inline float seed_rsqrt(float m)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(m));
    return y;
#else
    return 1.0f / sqrtf(m);
#endif
}

PLCG_HD inline float seed_rcp(float m)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(m));
    return y;
#else
    return 1.0f / m;
#endif
}

// m in [1, 4) to 23 bits of mantissa, from the bits of a double with biased
// exponent 1023 or 1024 (integer operations: conversions are FP64 instructions).
PLCG_HD inline float narrow_bits(uint64_t b)
{
    const uint32_t u = ((uint32_t)(b >> 52) - 1023u + 127u) << 23 | (uint32_t)(b >> 29 & 0x7fffffu);
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float f;
    memcpy(&f, &u, sizeof f);
    return f;
#endif
}

// The double of a positive normal float.
PLCG_HD inline double widen_bits(float f)
{
#ifdef __CUDA_ARCH__
    const uint32_t u = __float_as_uint(f);
#else
    uint32_t u;
    memcpy(&u, &f, sizeof u);
#endif
    return fx_from_bits(((uint64_t)u << 29) + (896ull << 52));
}

PLCG_HD PLCG_FX_NOINLINE static double plain_rsqrt(double x) { return 1.0 / sqrt(x); }
PLCG_HD PLCG_FX_NOINLINE static double plain_rcp(double x) { return 1.0 / x; }

// 1 / sqrt(m) from the seed y, m in [1, 4).
PLCG_HD inline double rsqrt_from_seed(double m, double y)
{
    const double e = fma(-m, y * y, 1.0);
    return fma(y * e, fma(e, fma(e, 0.3125, 0.375), 0.5), y);
}

// 1 / m from the seed y, m in [1, 2).
PLCG_HD inline double rcp_from_seed(double m, double y)
{
    const double e = fma(-m, y, 1.0);
    return fma(y, fma(fma(e, e, e), e, e), y);
}

PLCG_HD inline double fast_rsqrt(double x)
{
    const uint64_t b = fx_bits(x);
    const int ex = (int)(b >> 52);                   // with the sign: > 2046 for negative numbers
    if (__builtin_expect(ex < 1 || ex > 2046, 0)) return plain_rsqrt(x);
    // x = m 4^k, m in [1, 4)
    const int odd = (ex - 1023) & 1, k = (ex - 1023 - odd) / 2;
    const uint64_t mb = (b & 0xfffffffffffffull) | (uint64_t)(1023 + odd) << 52;
    const double r = rsqrt_from_seed(fx_from_bits(mb), widen_bits(seed_rsqrt(narrow_bits(mb))));
    return fx_from_bits(fx_bits(r) - ((uint64_t)(int64_t)k << 52));   // r 2^-k: normal
}

PLCG_HD inline double fast_rcp(double x)
{
    const uint64_t b = fx_bits(x);
    const int ex = (int)(b >> 52) & 0x7ff;
    if (__builtin_expect(ex < 1 || ex > 2044, 0)) return plain_rcp(x);
    const uint64_t mb = (b & 0xfffffffffffffull) | 1023ull << 52;
    const double r = rcp_from_seed(fx_from_bits(mb), widen_bits(seed_rcp(narrow_bits(mb))));   // in (1/2, 1]
    return fx_from_bits((fx_bits(r) - ((uint64_t)(int64_t)(ex - 1023) << 52)) | (b & 1ull << 63));
}

}  // namespace plcg
