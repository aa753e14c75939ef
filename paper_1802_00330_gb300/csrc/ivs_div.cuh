// ivs_div.cuh -- correctly rounded FP64 division on the integer pipes.
//
// The library's division runs on the FP64 pipe, which is the contraction's bottleneck: 1000
// cycles in a dependent chain and 7 (to nearest) to 12 (directed) adds' worth of its rate,
// against 361 cycles of the integer and FP32 pipes here (a test compares 2.3e8 pairs of
// operands with the library in the three roundings).  Contraction stage: n = 5 bisection 1.58 -> 1.47 ms, n = 6 solve 0.74 -> 0.71,
// kinema 87.9 -> 84.1, n = 8 of the 64-system batch 128.8 -> 123.6.  2n
// divisions follow one another in a box's sweep.  This one is a digit recurrence of very high
// radix (Ercegovac and Lang, Division and Square Root, 1994): signed digits of 17-18 bits,
// each estimated in single precision from the remainder's leading bits and the divisor's
// reciprocal and multiplied back exactly in 64-bit integers, so the quotient's 53 bits take
// three digits and the final remainder decides the rounding.  It has no constants beyond the
// format's.
//
// Digit error: the divisor's top 32 bits as a float and its approximate reciprocal are within
// 2^-22.3 (relative), the remainder's float within 2^-24 and its truncation within 2^-29 of
// the divisor; a digit is below 2^19, so it is off by at most 2^-2.9 + 1/2 and the next
// remainder stays below 0.64 divisors in magnitude: the digits never overflow, and one
// conditional correction makes the last remainder non-negative.
#pragma once
#include <cstdint>

namespace ivs {

enum : int { DIV_RN, DIV_RD, DIV_RU };

template <int MODE>
__device__ __forceinline__ double div_library(double a, double b) {
    if (MODE == DIV_RD) return __ddiv_rd(a, b);
    if (MODE == DIV_RU) return __ddiv_ru(a, b);
    return __ddiv_rn(a, b);
}

__device__ __forceinline__ float rcp_approx(float x) {
#ifdef __CUDA_ARCH__
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
#else
    return 1.0f / x;   // compiled for the host by a test
#endif
}

// a / b rounded to nearest even (DIV_RN), down (DIV_RD) or up (DIV_RU): the library's value for
// every pair of operands.  Zeros divided by normal numbers are handled here (the eliminated
// columns are full of them); subnormal, infinite or NaN operands, zero divisors and quotients
// near the ends of the exponent range go to the library.
template <int MODE>
__device__ __forceinline__ double div_exact(double a, double b) {
    const uint64_t ua = (uint64_t)__double_as_longlong(a), ub = (uint64_t)__double_as_longlong(b);
    const int ea = (int)(ua >> 52) & 0x7FF, eb = (int)(ub >> 52) & 0x7FF;
    const uint64_t sign = (ua ^ ub) & 0x8000000000000000ull;
    const uint64_t frac = 0x000FFFFFFFFFFFFFull, one = 0x0010000000000000ull;
    const bool bn = (unsigned)(eb - 1) < 2046u;
    if (bn && (ua << 1) == 0) return __longlong_as_double((long long)sign);
    int e = ea - eb + 1023;
    if (!(bn && (unsigned)(ea - 1) < 2046u && e > 1 && e < 2046)) return div_library<MODE>(a, b);
    const int64_t mb = (int64_t)((ub & frac) | one);
    int64_t r = (int64_t)((ua & frac) | one);
    if (r < mb) {   // quotient in [1, 2)
        r <<= 1;
        e -= 1;
    }
    // scale: remainder / 2^23 and divisor / 2^21 as floats, digits of 2^18, 2^17, 2^17.  The products
    // reach 2^72 and their differences stay below 2^53, so they are taken modulo 2^64.
    const float inv = rcp_approx(__uint2float_rn((uint32_t)(mb >> 21))) * 0x1p+20f;   // 2^(23 - 21 + 18)
    const int d1 = __float2int_rn(__int2float_rn((int)(r >> 23)) * inv);
    r = (int64_t)(((uint64_t)r << 18) - (uint64_t)(int64_t)d1 * (uint64_t)mb);
    const float inv2 = inv * 0.5f;
    const int d2 = __float2int_rn(__int2float_rn((int)(r >> 23)) * inv2);
    r = (int64_t)(((uint64_t)r << 17) - (uint64_t)(int64_t)d2 * (uint64_t)mb);
    const int d3 = __float2int_rn(__int2float_rn((int)(r >> 23)) * inv2);
    r = (int64_t)(((uint64_t)r << 17) - (uint64_t)(int64_t)d3 * (uint64_t)mb);
    int64_t q = ((((int64_t)d1 << 17) + d2) << 17) + d3;
    if (r < 0) {
        q -= 1;
        r += mb;
    }
    // q = floor of the quotient times 2^52, r the remainder
    bool up;
    if (MODE == DIV_RN) up = 2 * r > mb || (2 * r == mb && (q & 1));
    else up = r != 0 && (MODE == DIV_RU) == (sign == 0);
    const uint64_t bits = ((uint64_t)e << 52) + (uint64_t)(q - (int64_t)one) + (up ? 1u : 0u);
    return __longlong_as_double((long long)(bits | sign));
}

}  // namespace ivs
