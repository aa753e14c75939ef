// Operands for the tests of ivs_div.cuh, host and device: item i of class k.  Classes: 0 any
// exponents, 1 exponents near each other, 2 exact quotients, 3 one unit beside exact quotients, 4
// quotients beside the middle of two doubles, 5 quotients at the ends of the exponent range, 6
// zeros, subnormals, infinities and NaN in all pairs with ordinary numbers.
#pragma once
#include <cstdint>

enum { kClasses = 7 };

IVS_HD inline uint64_t mix(uint64_t x) {   // splitmix64 (Steele, Lea and Flood 2014)
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}
IVS_HD inline uint64_t number(uint64_t sign, uint64_t exponent, uint64_t fraction) {
    return (sign << 63) | (exponent << 52) | (fraction & 0x000FFFFFFFFFFFFFull);
}
IVS_HD inline uint64_t special(uint64_t r) {
    switch (r % 8) {
        case 0: return 0;
        case 1: return number(0, 0, mix(r));                     // subnormal
        case 2: return number(0, 0, 1);
        case 3: return number(0, 2047, 0);                       // infinity
        case 4: return number(0, 2047, 1ull << 51);              // NaN
        case 5: return number(0, 1, 0);
        case 6: return number(0, 2046, ~0ull);
        default: return number(0, 1 + mix(r) % 2046, mix(r + 1));
    }
}
IVS_HD inline void operands(int k, uint64_t i, uint64_t &a, uint64_t &b) {
    const uint64_t r = mix(i * 8 + (uint64_t)k), s = mix(r), t = mix(s);
    const uint64_t sa = r >> 63, sb = s >> 63;
    if (k == 0) {
        a = number(sa, 1 + r % 2046, s);
        b = number(sb, 1 + s % 2046, t);
        return;
    }
    if (k == 1 || k == 5) {
        // the quotient's exponent: near 1, or from subnormal to overflow within 4 of the ends
        const int64_t d = k == 1 ? (int64_t)(t % 8) - 4 : (t & 1) ? 1020 + (int64_t)(t / 2 % 8) : -1026 + (int64_t)(t / 2 % 8);
        const int64_t eb = d > 0 ? 1 + (int64_t)(r % 3) : 2046 - (int64_t)(r % 3);
        const int64_t mid = 1023 + (int64_t)(r % 64);
        const int64_t ea = k == 1 ? mid + d : eb + d;
        const int64_t ee = k == 1 ? mid : eb;
        a = number(sa, (uint64_t)(ea < 1 ? 1 : ea > 2046 ? 2046 : ea), s);
        b = number(sb, (uint64_t)ee, (t & 2) ? t : 0);
        return;
    }
    if (k == 6) {
        a = special(r % 64 / 8) | (sa << 63);
        b = special(r % 8) | (sb << 63);
        return;
    }
    uint64_t x, y;
    if (k == 4) {
        // an odd b of 53 bits and an odd Q of 54 with b Q = a 2^54 + 1 or - 1: a / b is the middle Q / 2^54 of two
        // doubles to within 2^-106
        y = (s >> 12) | (1ull << 52) | 1ull;
        uint64_t inv = y;   // the inverse of b modulo 2^64, by Newton's steps (3, 6, ... 96 bits)
        for (int n = 0; n < 5; n++) inv *= 2 - y * inv;
        uint64_t q = inv & ((1ull << 54) - 1);
        const bool minus = !(q >> 53);
        if (minus) q = (1ull << 54) - q;
        const uint64_t y0 = y & 0xFFFFFFFFull, y1 = y >> 32, q0 = q & 0xFFFFFFFFull, q1 = q >> 32;
        const uint64_t mid = y1 * q0 + ((y0 * q0) >> 32), mid2 = y0 * q1 + (mid & 0xFFFFFFFFull);
        const uint64_t hi = y1 * q1 + (mid >> 32) + (mid2 >> 32), lo = y * q;
        x = ((hi << 10) | (lo >> 54)) + (minus ? 1 : 0);
    } else {
        // 2, 3: a = q b with q of w and b of 53 - w bits
        const int w = 1 + (int)(s % 52);
        y = ((t >> 11) >> w) | 1ull;
        x = ((r >> 11) >> (53 - w)) * y;
        if (x == 0) x = 1;
    }
    union { double d; uint64_t u; } da, db;
    da.d = (double)x;
    db.d = (double)y;
    a = da.u | (sa << 63);
    b = db.u | (sb << 63);
    if (k == 3) a = (t & 1) ? a + 1 : a - 1;
}
