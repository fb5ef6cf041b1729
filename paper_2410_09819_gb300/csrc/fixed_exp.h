// Square root, division by a fixed number and e^-x of FP64 numbers in 64-bit integer arithmetic.
//
// GB300 retires 1.7 FP64 operations a clock and SM against about 60 integer ones (20 multiply-adds
// of 32 x 32 + 64 bits), and an FP64 square root, division and exponential are software sequences of
// 10, 7 and 16 FP64 operations: the Matern generator spends 35 of its 42 FP64 operations on them.
// Here the square root and the quotient are the correctly rounded ones (the same bits as IEEE
// arithmetic) and e^-x is within 0.52 units in the last place for x < 40 and 0.62 for x < 700.  Methods: Newton's iteration on an
// FP32 reciprocal square root, a reciprocal prepared once, and 2^-u = 2^-n 2^-(i/1024) e^-z with a
// table over i and the Taylor series of e^-z for z < 2^-10.5 ln 2.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#ifndef FIXED_FN
#define FIXED_FN __device__ __forceinline__
#endif

namespace tc {
namespace fx {

#ifdef __CUDA_ARCH__
FIXED_FN uint64_t mulhi(uint64_t a, uint64_t b) { return __umul64hi(a, b); }
FIXED_FN int64_t mulhi_s(int64_t a, int64_t b) { return __mul64hi(a, b); }
FIXED_FN uint32_t mulhi32(uint32_t a, uint32_t b) { return __umulhi(a, b); }
FIXED_FN float rsqrt_f(float x) { return rsqrtf(x); }
FIXED_FN uint32_t to_u32(float x) { return __float2uint_rz(x); }          // saturates
FIXED_FN uint64_t bits(double x) { return (uint64_t)__double_as_longlong(x); }
FIXED_FN double from_bits(uint64_t w) { return __longlong_as_double((long long)w); }
#else                                                // the same arithmetic for tests on the CPU
FIXED_FN uint64_t mulhi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
FIXED_FN int64_t mulhi_s(int64_t a, int64_t b) { return (int64_t)(((__int128)a * b) >> 64); }
FIXED_FN uint32_t mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
FIXED_FN float rsqrt_f(float x) { return 1.0f / sqrtf(x); }
FIXED_FN uint32_t to_u32(float x) { return x >= 4294967296.0f ? 0xFFFFFFFFu : (uint32_t)x; }
FIXED_FN uint64_t bits(double x) { uint64_t w; memcpy(&w, &x, 8); return w; }
FIXED_FN double from_bits(uint64_t w) { double x; memcpy(&x, &w, 8); return x; }
#endif

// A positive number m 2^e, m in [2^52, 2^53).
struct Num {
    uint64_t m;
    int e;
};

// RN(sqrt(s)) of a positive normal number.  With m in [2^52, 2^54) and an even exponent,
// P = m Y 2^-22 with Y = 2^47 / sqrt(m 2^-22) to 21 bits; P Y 2^-32 = 2^62 (1 - e), and
// W = P (1 + e/2 + 3e^2/8) = sqrt(m) 2^36 to a few units, ten bits more than the result has.  Where
// those ten bits leave the rounding open (one argument in 64), the square of the boundary decides.
FIXED_FN Num sqrt_rn(double s) {
    const uint64_t w = bits(s);
    int e = (int)(w >> 52) - 1075;
    uint64_t m = (w & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    if (e & 1) {
        m <<= 1;
        --e;
    }
    const uint32_t Y = to_u32(rsqrt_f((float)(uint32_t)(m >> 22)) * 140737488355328.0f);    // 2^47
    const uint64_t A = m << 10;
    const uint64_t P = (A >> 32) * Y + (((A & 0xFFFFFFFFull) * Y) >> 32);
    const uint64_t Q = (P >> 32) * Y + (((P & 0xFFFFFFFFull) * Y) >> 32);
    const int64_t E = (int64_t)((1ull << 62) - Q);
    const int64_t E21 = E >> 21;
    const int64_t E2 = (E >> 1) + ((((E21 * E21) >> 20) * 3) >> 3);
    const uint64_t W = P + (uint64_t)(mulhi_s((int64_t)(P >> 1), E2 << 20) >> 17);
    uint64_t h = (W + 512) >> 10;
    const int low = (int)(W & 1023);
    if (low >= 496 && low < 528) {
        const uint64_t t = 2 * (W >> 10) + 1;           // the boundary, and its distance modulo 2^64
        h = (W >> 10) + ((int64_t)((m << 54) - t * t) > 0 ? 1 : 0);
    }
    e = e / 2 - 26;                                     // sqrt(s) = W 2^-36 2^(e/2), h = W 2^-10
    if (h >> 53) {
        h >>= 1;
        ++e;
    }
    return {h, e};
}

// RN(sqrt(s)) and RN(1 / RN(sqrt(s))) of a positive normal number together: the correction that turns
// W into a square root turns Y into its reciprocal as well, R = 2^89 / sqrt(m); what rounding adds to
// the root then moves the reciprocal by R^2 2^-125 times as much.
FIXED_FN void sqrt_recip_rn(double s, Num &root, Num &recip) {
    const uint64_t w = bits(s);
    int e = (int)(w >> 52) - 1075;
    uint64_t m = (w & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    if (e & 1) {
        m <<= 1;
        --e;
    }
    const uint32_t Y = to_u32(rsqrt_f((float)(uint32_t)(m >> 22)) * 140737488355328.0f);    // 2^47
    const uint64_t A = m << 10;
    const uint64_t P = (A >> 32) * Y + (((A & 0xFFFFFFFFull) * Y) >> 32);
    const uint64_t Q = (P >> 32) * Y + (((P & 0xFFFFFFFFull) * Y) >> 32);
    const int64_t E = (int64_t)((1ull << 62) - Q);
    const int32_t E21 = (int32_t)(E >> 21);
    const int64_t E2 = (E >> 1) + (((((int64_t)E21 * E21) >> 20) * 3) >> 3);
    const uint64_t W = P + (uint64_t)(mulhi_s((int64_t)(P >> 1), E2 << 20) >> 17);
    const uint64_t R = ((uint64_t)Y << 31) + (uint64_t)mulhi_s((int64_t)((uint64_t)Y << 31), E2 << 2);
    const uint32_t S = (uint32_t)(((R >> 32) * (R >> 32)) >> 31);
    uint64_t h = (W + 512) >> 10;
    const int low = (int)(W & 1023);
    if (low >= 496 && low < 528) {
        const uint64_t t = 2 * (W >> 10) + 1;           // the boundary, and its distance modulo 2^64
        h = (W >> 10) + ((int64_t)((m << 54) - t * t) > 0 ? 1 : 0);
    }
    const uint64_t V = R - (uint64_t)(((int64_t)S * (int32_t)((h << 10) - W)) >> 30);
    e = e / 2 - 26;                                     // sqrt(s) = W 2^-36 2^(e/2), h = W 2^-10
    if (h >> 53) {
        h >>= 1;
        ++e;
    }
    root = {h, e};
    uint64_t q = (V >> 10) + ((V >> 9) & 1);
    const int lowv = (int)(V & 1023);
    if (lowv >= 496 && lowv < 528) {
        const uint64_t t = 2 * (V >> 10) + 1;           // t h against 2^106, modulo 2^64
        q = (V >> 10) + ((int64_t)(0 - t * h) > 0 ? 1 : 0);
    }
    int er = -105 - e;
    if (q >> 53) {
        q >>= 1;
        ++er;
    }
    if (h == 1ull << 52) {
        q = 1ull << 52;
        er = -104 - e;
    }
    recip = {q, er};
}

// Division by a fixed a = m 2^e: v = floor(2^116 / m), at most 2^64 - 1.
struct Divisor {
    uint64_t m, v;
    int e;
};
// (not on the hot path: one division by repeated halving)
FIXED_FN Divisor make_divisor(double a) {
    const uint64_t w = bits(a);
    Divisor d;
    d.e = (int)(w >> 52) - 1075;
    d.m = (w & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    uint64_t rem = 1ull << 52, q = 0;                   // 2^116 = 2^52 2^64: 64 quotient bits after rem / m
    const bool one = rem >= d.m;                        // m = 2^52: the quotient is 2^64
    for (int i = 0; i < 64; ++i) {
        rem <<= 1;
        q <<= 1;
        if (rem >= d.m) {
            rem -= d.m;
            q |= 1;
        }
    }
    d.v = one ? ~0ull : q;
    return d;
}
// RN(h / a), by the prepared reciprocal; an open rounding (one argument in 64) is decided by the
// remainder of the boundary.
FIXED_FN Num div_rn(const Num &h, const Divisor &a) {
    uint64_t Q = mulhi(h.m << 11, a.v);                 // (h / m) 2^63
    int k = 53, e = h.e - a.e - 52;
    if (!(Q >> 63)) {
        Q <<= 1;
        k = 54;
        --e;
    }
    uint64_t q = (Q >> 11) + ((Q >> 10) & 1);
    const int low = (int)(Q & 2047);
    if (low >= 1008 && low < 1040) {
        const uint64_t t = 2 * (Q >> 11) + 1;
        q = (Q >> 11) + ((int64_t)((h.m << k) - t * a.m) > 0 ? 1 : 0);
    }
    if (q >> 53) {
        q >>= 1;
        ++e;
    }
    return {q, e};
}
FIXED_FN double value(const Num &x) { return from_bits(((uint64_t)(x.e + 1075) << 52) | (x.m & 0xFFFFFFFFFFFFFull)); }

constexpr int EXP_TABLE = 1024;
// Entry i of the table: 2^63 2^(-i / 1024), as a product over the bits of i of
// 2^64 2^(-2^k / 1024), k = 0 .. 9.
FIXED_FN uint64_t exp_entry(int i) {
    constexpr uint64_t c[10] = {0xffd3a751c0f7e10cull, 0xffa756521c8daed2ull, 0xff4ecb59511ec8a5ull, 0xfe9e115c7b8f884cull,
                                0xfd3e0c0cf486c175ull, 0xfa83b2db722a033aull, 0xf5257d152486cc2cull, 0xeac0c6e7dd24392full,
                                0xd744fccad69d6af4ull, 0xb504f333f9de6484ull};
    uint64_t t = 1ull << 63;
    for (int k = 0; k < 10; ++k)
        if ((i >> k) & 1) t = mulhi(t, c[k]);
    return t;
}

// e^-x for 0 < x < 700
FIXED_FN double exp_neg(const Num &x, const uint64_t *table) {
    // u = x log2(e) = (hi : lo) 2^(p - 126), p the exponent of x's leading bit
    const int p = x.e + 52;
    const uint64_t X = x.m << 11, L = 0xb8aa3b295c17f0bcull;      // 2^63 log2(e)
    const uint64_t hi = mulhi(X, L), lo = X * L;
    const int s = 62 - p;                               // binary digits of hi below the point: 53 ..
    int n = 0;
    uint64_t f;                                         // fraction, 64 bits
    if (s < 64) {
        n = (int)(hi >> s);
        f = (hi << (64 - s)) | (lo >> s);
    } else {
        f = s < 128 ? hi >> (s - 64) : 0;
    }
    // 2^-f = T[i] e^-z, z = f' ln 2 with f' < 2^-10: Z = z 2^74
    const uint64_t T = table[f >> 54], Z = mulhi(f << 10, 0xb17217f7d1cf79acull);
    const uint64_t Z2 = mulhi(Z, Z);                    // z^2 2^84
    const uint32_t zs = (uint32_t)(Z >> 32), c3 = mulhi32((uint32_t)(Z2 >> 32), zs);      // z^3 2^62
    uint64_t q = ((uint64_t)c3 * 0xAAAAAAABull) >> 22;  // z^3 / 6 2^74
    q -= ((q >> 20) * zs) >> 24;                        // (1 - z / 4)
    const uint64_t Wz = Z - (Z2 >> 11) + q;             // (1 - e^-z) 2^74
    const uint64_t R = T - (mulhi(T, Wz) >> 10);        // 2^63 2^-f, in (2^62, 2^63]
    if (R >> 63) return from_bits((uint64_t)(1023 - n) << 52);
    const uint64_t mant = (R + 512) >> 10;              // 53 bits, or 2^53
    return from_bits(((uint64_t)(1022 - n) << 52) + (mant - (1ull << 52)));
}

}  // namespace fx
}  // namespace tc
