// FP64 products of 64 x 64 blocks on warp-level FP16 MMAs, for products too small for the
// tile-sized tensor-core kernel (k_ozaki.cu): the inverse of a diagonal tile of an all-FP64 map, and
// of any map out of core (mixed maps in core take k_trinv_batched, see there).
//
// The arithmetic is that of k_ozaki.cu (seven base-256 digits of an operand in FP16, 28 digit
// products s + t <= 6 with exact FP32 sums, integer recombination), but with an exponent of its
// own for every row of X and of Y^T instead of one for a tile: X Y^T is taken in steps of 64 along
// K, and in each step row r of an operand is rounded to 2^-57 of its largest entry there.  One step
// of one block is 3584 mma.sync.m16n8k16 on one SM.
//
// Why: an SM retires 1.7 FP64 multiply-adds a clock, so a 64 x 64 x 64 step on the FP64 pipe takes
// 69 us on its SM; mma.sync runs 1010 FP16 multiply-adds a clock (measured), so the 28 digit
// products take 3.5 us, and the conversions about as long.
//
// Infinities and NaNs: a row (column) that holds one makes its row (column) of the product NaN.
#include "digits.h"
#include "tc_internal.h"

#include <cuda_fp16.h>

namespace tc {
namespace bg {

constexpr int B = 64;                      // block size and K step
constexpr int NP = 7;                      // digit planes
constexpr int RS = 72;                     // halves per plane row: 144 bytes, conflict-free for the fragment loads
constexpr int PLANE = B * RS;              // halves of one plane
constexpr int BAD = 1 << 20;               // exponent of a row with an infinity or a NaN
constexpr size_t SMEM = (size_t)2 * NP * PLANE * sizeof(__half) + (2 * 4 * B + 2 * B) * sizeof(int);

// An operand block: element (r, k) at p[r * rs + k * ks].
struct Op {
    const double *p;
    int64_t rs, ks;
};

// 16 elements of row r (thread (r, kq), K range 16 kq ...) and the largest exponent among them
__device__ __forceinline__ void load16(const Op &o, int r, int kq, double (&x)[16], int *emax) {
    const double *p = o.p + (int64_t)r * o.rs + (int64_t)(16 * kq) * o.ks;
    int m = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = p[(int64_t)i * o.ks];
#pragma unroll
    for (int i = 0; i < 16; ++i) m = max(m, (__double2hiint(x[i]) >> 20) & 0x7FF);
    emax[kq * B + r] = m;
}
__device__ __forceinline__ void planes16(const double (&x)[16], int e, int r, int kq, __half *P) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        long long q[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) q[u] = fixed56(x[8 * h + u], e);
        uint32_t lo[8], hi[8];
        biased8(q, lo, hi);
#pragma unroll
        for (int s = 0; s < NP; ++s)
            *reinterpret_cast<uint4 *>(P + s * PLANE + r * RS + 16 * kq + 8 * h) = digit8(lo, hi, s);
    }
}
// row exponent from the four partial maxima: |x| < 2^e (all zero: any), BAD with an inf or a NaN
__device__ __forceinline__ int row_exp(const int *emax, int r) {
    const int m = max(max(emax[r], emax[B + r]), max(emax[2 * B + r], emax[3 * B + r]));
    return m == 0x7FF ? BAD : max(m, 1) - 1022;
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// t 2^e rounded to FP64 with integer operations (a 64-bit conversion runs on the FP64 pipe)
__device__ __forceinline__ double scaled(long long t, int e) {
    if (t == 0) return 0.0;
    const unsigned long long u = t < 0 ? (unsigned long long)(-t) : (unsigned long long)t;
    const int lz = __clzll((long long)u);
    unsigned long long m = u << lz;                    // leading bit at 63
    int ex = 63 - lz + e + 1023;
    m += 0x400;                                        // round to 53 bits
    if (m < 0x400) {                                   // carried out of bit 63
        m = 1ull << 63;
        ++ex;
    }
    if (ex <= 0 || ex >= 0x7FF) return ldexp((double)t, e);
    const unsigned long long w = ((unsigned long long)ex << 52) | ((m >> 11) & 0xFFFFFFFFFFFFFull);
    return __longlong_as_double((long long)(t < 0 ? w | (1ull << 63) : w));
}

// One step: acc (16 elements a thread, in the fragment layout) += X Y^T over 64 elements of K.
// 256 threads; warp w owns rows 16 (w & 3) .. and columns 32 (w >> 2) .. of the block.  K rows are contiguous in memory for an operand with
// ks == 1, rows of the block otherwise: threads are laid out for coalesced loads either way.
__device__ __forceinline__ void step(const Op &X, const Op &Y, double (&acc)[16], uint8_t *smem) {
    __half *PX = reinterpret_cast<__half *>(smem), *PY = PX + NP * PLANE;
    int *ex4 = reinterpret_cast<int *>(smem + (size_t)2 * NP * PLANE * sizeof(__half)), *ey4 = ex4 + 4 * B;
    int *ex = ey4 + 4 * B, *ey = ex + B;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rx = X.ks == 1 ? tid >> 2 : tid & 63, kx = X.ks == 1 ? tid & 3 : tid >> 6;
    const int ry = Y.ks == 1 ? tid >> 2 : tid & 63, ky = Y.ks == 1 ? tid & 3 : tid >> 6;
    __syncthreads();                                   // the previous step's fragments are read
    double x[16], y[16];
    load16(X, rx, kx, x, ex4);
    load16(Y, ry, ky, y, ey4);
    __syncthreads();
    {
        const int e = row_exp(ex4, rx);
        if (kx == 0) ex[rx] = e;
        planes16(x, e == BAD ? 0 : e, rx, kx, PX);
    }
    {
        const int e = row_exp(ey4, ry);
        if (ky == 0) ey[ry] = e;
        planes16(y, e == BAD ? 0 : e, ry, ky, PY);
    }
    __syncthreads();
    const int g = lane >> 2, t = lane & 3, r0 = 16 * (warp & 3), c0 = 32 * (warp >> 2);
    float d[NP][4][4];
#pragma unroll
    for (int s = 0; s < NP; ++s)
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) d[s][n][i] = 0.f;
#pragma unroll 1
    for (int ks = 0; ks < 4; ++ks) {
        uint32_t a[NP][4];
        const __half *pa = PX + (r0 + g) * RS + 16 * ks + 2 * t;
#pragma unroll
        for (int s = 0; s < NP; ++s) {
            a[s][0] = *reinterpret_cast<const uint32_t *>(pa + s * PLANE);
            a[s][1] = *reinterpret_cast<const uint32_t *>(pa + s * PLANE + 8 * RS);
            a[s][2] = *reinterpret_cast<const uint32_t *>(pa + s * PLANE + 8);
            a[s][3] = *reinterpret_cast<const uint32_t *>(pa + s * PLANE + 8 * RS + 8);
        }
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const __half *pb = PY + (c0 + 8 * n + g) * RS + 16 * ks + 2 * t;
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                uint32_t bq[2];
                bq[0] = *reinterpret_cast<const uint32_t *>(pb + q * PLANE);
                bq[1] = *reinterpret_cast<const uint32_t *>(pb + q * PLANE + 8);
#pragma unroll
                for (int s = 0; s + q < NP; ++s) mma16816(d[s + q][n], a[s], bq);
            }
        }
    }
    // group sums are integers of at most 2.25 x 2^22: sum = 2^(ex + ey - 56) t
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            long long hi = 0, lo = 0;
#pragma unroll
            for (int s = 0; s < 4; ++s) hi += (long long)__float2int_rn(d[s][n][i]) * (1 << (8 * (3 - s)));
#pragma unroll
            for (int s = 4; s < NP; ++s) lo += (long long)__float2int_rn(d[s][n][i]) * (1 << (8 * (6 - s)));
            const int er = ex[r0 + g + 8 * (i >> 1)], ec = ey[c0 + 8 * n + 2 * t + (i & 1)];
            const double v = (er == BAD || ec == BAD) ? __longlong_as_double(0x7FF8000000000000ll)
                                                      : scaled(hi * 65536 + (lo >> 8), er + ec - 56);
            acc[4 * n + i] += v;
        }
}
// row and column of element i of a thread's fragment
__device__ __forceinline__ int frag_row(int i) { return 16 * ((threadIdx.x >> 5) & 3) + ((threadIdx.x & 31) >> 2) + 8 * ((i >> 1) & 1); }
__device__ __forceinline__ int frag_col(int i) { return 32 * (threadIdx.x >> 7) + 8 * (i >> 2) + 2 * (threadIdx.x & 3) + (i & 1); }

}  // namespace bg

// ------------------------------------------------------------ inverse of a diagonal tile
// Y = L^{-1} for a lower-triangular b x b tile (column-major): the 64 x 64 diagonal blocks by
// substitution, then by doubling, [L11 0; L21 L22]^{-1} = [I11 0; -I22 (L21 I11) I22], with the two
// products of a level as block products (T = L21 I11 waits in Y's upper part, block (r, c) in the
// place of its transpose, and the part is cleared at the end).  Column by column on the FP64 pipe the inverse of a 1024 tile took 1.13 ms and that of
// a 2048 tile 4.25 ms.

// Diagonal blocks: L y_c = e_c with M = diag(1 / l_rr) L, a warp per column, lane l holding rows l
// and l + 32: step j is a shuffle and a multiply-add.  blockIdx.y takes 16 of the 64 columns.
__global__ void __launch_bounds__(256) k_trinv64(const TEntry *__restrict__ e, TEntry one, int b) {
    __shared__ double M[64][65], rinv[64];       // M[j][r] = l_rj / l_rr, r > j
    const TEntry E = e ? e[blockIdx.z] : one;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t o = (int64_t)blockIdx.x * 64 * (b + 1);
    for (int idx = tid; idx < 4096; idx += 256) {
        const int r = idx & 63, c = idx >> 6;
        if (r >= c) M[c][r] = E.L[o + (int64_t)c * b + r];
    }
    __syncthreads();
    if (tid < 64) rinv[tid] = 1.0 / M[tid][tid];
    __syncthreads();
    for (int j = warp; j < 64; j += 8) {
        if (j < 31 && lane > j) M[j][lane] *= rinv[lane];
        if (lane + 32 > j) M[j][lane + 32] *= rinv[lane + 32];
    }
    __syncthreads();
    for (int q = 0; q < 2; ++q) {
        const int c = (int)blockIdx.y + 4 * (warp + 8 * q);      // columns of long and short chains mixed
        double y0 = lane == c ? rinv[lane] : 0.0, y1 = lane + 32 == c ? rinv[lane + 32] : 0.0;
#pragma unroll 4
        for (int j = c; j < 32; ++j) {
            const double yj = __shfl_sync(0xffffffffu, y0, j);
            if (lane > j) y0 = fma(-yj, M[j][lane], y0);
            y1 = fma(-yj, M[j][lane + 32], y1);
        }
#pragma unroll 4
        for (int j = c < 32 ? 0 : c - 32; j < 32; ++j) {
            const double yj = __shfl_sync(0xffffffffu, y1, j);
            if (lane > j) y1 = fma(-yj, M[j + 32][lane + 32], y1);
        }
        E.Y[o + (int64_t)c * b + lane] = y0;
        E.Y[o + (int64_t)c * b + lane + 32] = y1;
    }
}

// One product of a doubling level: pairs of s and up to s blocks, block (rb, cb) of the product of
// pair p.  phase 0: T = L21 I11 (K blocks cb .. s - 1), block (rb, cb) into Y's block (cb, rb) above
// the diagonal; phase 1: I21 = -I22 T (K blocks 0 .. rb).  Blocks with the longest sums come first.
__global__ void __launch_bounds__(256, 1)
k_trinv_level(const TEntry *__restrict__ e, TEntry one, int b, int s, int phase) {
    extern __shared__ __align__(16) uint8_t bsm[];
    const TEntry E = e ? e[blockIdx.z] : one;
    const int nb = b / 64, o = (int)blockIdx.y * 2 * s, s2 = min(s, nb - o - s);   // second half: s2 blocks
    const int a = (int)blockIdx.x / s, c = (int)blockIdx.x % s;
    const int rb = phase ? s - 1 - a : c, cb = phase ? c : a;
    if (rb >= s2) return;
    const int64_t r0 = (int64_t)(o + s + rb) * 64, c0 = (int64_t)(o + cb) * 64;
    double acc[16] = {};
    for (int kb = phase ? 0 : cb; kb < (phase ? rb + 1 : s); ++kb) {
        if (phase == 0) {
            const int64_t k0 = (int64_t)(o + kb) * 64;
            bg::step({E.L + k0 * b + r0, 1, b}, {E.Y + c0 * b + k0, b, 1}, acc, bsm);
        } else {
            const int64_t k0 = (int64_t)(o + s + kb) * 64;
            bg::step({E.Y + k0 * b + r0, 1, b}, {E.Y + k0 * b + c0, b, 1}, acc, bsm);
        }
    }
    double *out = phase ? E.Y + c0 * b + r0 : E.Y + r0 * b + c0;
#pragma unroll
    for (int i = 0; i < 16; ++i) out[(int64_t)bg::frag_col(i) * b + bg::frag_row(i)] = phase ? -acc[i] : acc[i];
}
// zero the blocks above the diagonal blocks
__global__ void k_zero_above(const TEntry *__restrict__ e, TEntry one, int b) {
    const TEntry E = e ? e[blockIdx.z] : one;
    const int cb = (int)blockIdx.x + 1;
    for (int c = blockIdx.y; c < 64; c += gridDim.y)
        for (int r = threadIdx.x; r < cb * 64; r += blockDim.x) E.Y[((int64_t)cb * 64 + c) * b + r] = 0.0;
}

template <class K>
static void bg_smem(K *kernel, std::atomic<unsigned long long> &attr) {
    if (attrs_pending(attr)) {
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bg::SMEM);
        mark_attrs_set(attr);
    }
}
// Y = L^{-1} of n tiles (entries e on the device, or the one given by value)
static void trinv_launches(const TEntry *e, const TEntry &one, int n, int b, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    bg_smem(k_trinv_level, attr);
    const int nb = b / 64;
    k_trinv64<<<dim3(nb, 4, n), 256, 0, s>>>(e, one, b);
    for (int h = 1; h < nb; h *= 2) {
        const dim3 grid(h * h, (nb + h - 1) / (2 * h), n);     // pairs whose second half is not empty
        k_trinv_level<<<grid, 256, bg::SMEM, s>>>(e, one, b, h, 0);
        k_trinv_level<<<grid, 256, bg::SMEM, s>>>(e, one, b, h, 1);
    }
    if (nb > 1) k_zero_above<<<dim3(nb - 1, 16, n), 256, 0, s>>>(e, one, b);
}
void launch_trinv_batched(const TEntry *e, int n, int b, cudaStream_t s) {
    for (int i = 0; i < n; i += 65535) trinv_launches(e + i, TEntry{}, n - i < 65535 ? n - i : 65535, b, s);
}
void launch_trinv(const double *L, int b, double *Y, cudaStream_t s) { trinv_launches(nullptr, TEntry{L, Y}, 1, b, s); }

}  // namespace tc
