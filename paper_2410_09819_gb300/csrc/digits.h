// Base-256 digits of FP64 numbers in integer arithmetic (GB300 runs FP64 at 2 operations per clock
// per SM), shared by the digit-plane conversions (k_ozaki.cu) and the block products (k_bgemm.cu).
#pragma once
#include <cstdint>
#include <cuda_fp16.h>

namespace tc {

// q = x 2^(56 - e) rounded to the nearest integer from the bit pattern (|x| <= 2^e)
__device__ __forceinline__ long long fixed56(double x, int e) {
    const long long bits = __double_as_longlong(x);
    int ex = (int)((bits >> 52) & 0x7FF);
    long long m = bits & 0xFFFFFFFFFFFFFLL;
    if (ex == 0) ex = 1;                       // subnormal (or zero): no hidden bit
    else m |= 1LL << 52;                       // |x| = m 2^(ex - 1075)
    const int sh = ex - 1019 - e;              // x 2^(56 - e) = m 2^sh, sh <= 4
    long long q;
    if (sh >= 0) q = m << sh;
    else if (sh > -63) q = (m + (1LL << (-sh - 1))) >> (-sh);
    else q = 0;
    return bits < 0 ? -q : q;
}

// The seven base-256 digits of eight numbers as FP16, digit s of number u in half u of w[s].
// With the bias 0x80 in the six low bytes, byte 6 - s of q + bias is digit s plus 128, and what
// remains above them is the top digit, in [-256, 256].  A byte u under the exponent byte 0x64 is
// the FP16 number 1024 + u, and 1024 + u - 1152 the digit, exactly: a byte permute, a logic
// operation and a half2 subtraction make one digit of two numbers.
__device__ __forceinline__ uint4 digit8(const uint32_t (&lo)[8], const uint32_t (&hi)[8], int s) {
    uint32_t w[4];
    // 1024 + 128, and 1024 + 256 for the top digit
    const __half2 off = __half2half2(__ushort_as_half((unsigned short)(s == 0 ? 0x6500 : 0x6480)));
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        uint32_t h;
        if (s == 0) {                           // 256 + digit in 10 bits
            h = __byte_perm(hi[2 * v] + 0x01000000u, hi[2 * v + 1] + 0x01000000u, 0x7632u) | 0x64006400u;
        } else {
            const int byte = 6 - s;
            const uint32_t a = byte < 4 ? lo[2 * v] : hi[2 * v], c = byte < 4 ? lo[2 * v + 1] : hi[2 * v + 1];
            const uint32_t sel = (uint32_t)(byte & 3) | ((uint32_t)(4 + (byte & 3)) << 8);
            h = (__byte_perm(a, c, sel) & 0x00FF00FFu) | 0x64006400u;
        }
        const __half2 d = __hsub2(*reinterpret_cast<const __half2 *>(&h), off);
        w[v] = *reinterpret_cast<const uint32_t *>(&d);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// RN((2^24 hi + lo) 2^e) in integer arithmetic: two 64-bit conversions, a product and a multiply-add
// a value kept the FP64 pipe busy for 9000 cycles an item of k_zgemm.
__device__ __forceinline__ double fixed_sum(long long hi, long long lo, int e) {
    unsigned long long l = ((unsigned long long)hi << 24) + (unsigned long long)lo;
    long long h = (hi >> 40) + (lo >> 63) + (l < (unsigned long long)lo ? 1 : 0);
    const unsigned long long sign = (unsigned long long)h & (1ull << 63);
    if (sign) {
        l = 0 - l;
        h = ~h + (l == 0 ? 1 : 0);
    }
    if ((h | (long long)l) == 0) return 0.0;
    int x = 1022 + 127 + e;                             // biased exponent less one of a leading bit 127
    if (h == 0) {
        h = (long long)l;
        l = 0;
        x -= 64;
    }
    const int n = __clzll(h);
    x -= n;
    unsigned long long m = (unsigned long long)h << n;
    if (n) m |= l >> (64 - n);
    m |= (l << n) != 0 ? 1 : 0;                         // what lies below, for ties
    const unsigned long long q = (m >> 11) + (((m & 2047) + 1023 + ((m >> 11) & 1)) >> 11);
    if (x < 0 || x > 2044) return ldexp(sign ? -(double)q : (double)q, x - 1074);
    return __longlong_as_double((long long)(sign | (((unsigned long long)x << 52) + q)));
}
__device__ __forceinline__ void biased8(const long long (&q)[8], uint32_t (&lo)[8], uint32_t (&hi)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const unsigned long long n = (unsigned long long)q[u] + 0x0000808080808080ull;
        lo[u] = (uint32_t)n;
        hi[u] = (uint32_t)(n >> 32);
    }
}

}  // namespace tc
