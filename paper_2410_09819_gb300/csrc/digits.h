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
__device__ __forceinline__ void biased8(const long long (&q)[8], uint32_t (&lo)[8], uint32_t (&hi)[8]) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const unsigned long long n = (unsigned long long)q[u] + 0x0000808080808080ull;
        lo[u] = (uint32_t)n;
        hi[u] = (uint32_t)(n >> 32);
    }
}

}  // namespace tc
