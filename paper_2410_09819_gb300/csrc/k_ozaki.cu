// FP64 tile updates emulated on the FP16 tensor cores (GB300's FP64 pipe delivers only
// ~1.25 TFLOP/s; its FP16 tensor cores ~1.9 PFLOP/s).
//
// Splitting (the error-free slicing of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 2012, with a per-tile exponent):
// every final FP64 tile X with e = the smallest integer such that max|X| <= 2^e is written
// as X = 2^(e-8) sum_{s=0..6} 256^-s D_s + R with 7 integer "digit planes" D_s (D_0 in
// [-256, 256], the others in [-128, 127], |R| <= 2^(e-57)), each stored in FP16, which holds
// these integers exactly.  Then
//     X Y^T = 2^(ex+ey-16) sum_{g=0..6} 256^-g G_g,   G_g = sum_{s+t=g} D_s(X) D_t(Y)^T,
// dropping the pairs with s + t > 6 (six of weight 2^-72 and products below 2^14 each: 2^-55 of
// the product's scale at worst).  G_0 .. G_5 over 128 elements of K are integers of at most 2^24
// in magnitude, which the tensor cores' FP32 accumulation holds exactly (G_6 can pass 2^24 by an
// eighth, only where every digit is at its extreme; its last bit weighs 2^-64).  Every 128 elements
// the drain adds the group sums, shifted, to a fixed-point sum per element (two int64 words with a
// unit of 2^-64 of the largest source's scale), which becomes FP64 once, at the end.
// The result is the FP64 update up to FP64-level rounding relative to the tiles' scale
// (a normwise bound, which is what the factorization's backward error needs).
//
// Why base 256 in FP16: an exact product needs 28 plane pairs, against 105 for base 16 in E4M3
// (14 planes; the digits of base 256 do not fit E4M3), and the FP16 rate is half the E4M3 rate,
// so the same product takes 28 x 2 = 56 units of E4M3 work instead of 105.  The price is that the
// sums outgrow 24 bits after 128 elements of K, not a whole source tile, so TMEM is drained
// every 128 elements; the drain is integer work (a 32-bit conversion and a 64-bit multiply-add
// per value) and stays hidden behind the MMAs.
#include "digits.h"
#include "tc_internal.h"
#include "zgemm_common.h"

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <cstring>

namespace tc {

constexpr int ZS = ZF_PLANES;          // digit planes per tile
constexpr int ZBM = 128, ZBN = Z_BN;   // work item: 128 rows x 32 columns
constexpr int ZKB = 64;                // K bytes per stage
constexpr int ZKE = ZKB / 2;           //   = 32 FP16 elements (two MMAs of K = 16)
constexpr int ZFLUSH = 128;            // elements of K between two drains of the accumulators
constexpr int ZFB = ZFLUSH / ZKE;      //   = 4 stages
// Pipeline: a stage holds all X and Y planes of 32 elements of K (70 KB), so one barrier wait and
// one commit cover its 14 MMAs.  The MMA-issuing warp has to keep the tensor pipe fed, and every
// barrier wait in its stream costs 75-90 cycles: with X planes two to a stage of 64 elements and
// the Y planes in a ring of their own (10 waits per 128 elements of K instead of 4) the same work
// took 6400 cycles per 128 elements, with these stages 5950, and with the issue of a converged warp
// (zgemm_common.h) 4990 (measured).
constexpr int ZST = 3;                 // stages
constexpr int ZX_BYTES = ZBM * ZKB;    // 8 KB: one X plane block
constexpr int ZY_BYTES = ZBN * ZKB;    // 2 KB: one Y plane block
constexpr int ZSTAGE = ZS * (ZX_BYTES + ZY_BYTES);   // 70 KB: X planes, then Y planes
constexpr int ZDRAIN = 8;              // drain warps: two per TMEM lane quarter, 16 columns each
constexpr int ZTHREADS = 64 + 32 * ZDRAIN;   // producer, MMA, drain
constexpr unsigned long long ZLIMIT_NS = 4000000000ull;   // default bound of a pipeline wait
constexpr unsigned long long ZDRAIN_NS = 2000000000ull;   // bound of the teardown waits

// ------------------------------------------------------------------- digit planes
// Base-256 planes lie as the shared memory of k_zgemm wants them: columns in blocks of ZKE, in a block
// row after row of 64 bytes, the 16-byte pieces of a row in the order of the 64-byte swizzle
// (piece c of row r at c ^ (r / 2 mod 4)).  A stage's part of a plane is then one contiguous piece of 8
// or 2 KB, which a plain bulk copy brings at 117 bytes a clock and SM (95 on all SMs at once); boxes
// of 64-byte rows through a tensor map came at 60, a row a clock, however the rows lay.
__device__ __forceinline__ int64_t plane_at(int b, int row, int col) {      // element (row, col), col % 8 == 0
    return ((int64_t)(col / ZKE) * b + row) * ZKE + 8 * (((col % ZKE) / 8) ^ ((row >> 1) & 3));
}
// Base-256 planes of eight adjacent columns of a row (k_zgemm), one 16-byte store per plane.
__device__ __forceinline__ void put_planes8(const long long (&q)[8], __half *P, int64_t o, int64_t bb) {
    uint32_t lo[8], hi[8];
    biased8(q, lo, hi);
#pragma unroll
    for (int s = 0; s < ZS; ++s) *reinterpret_cast<uint4 *>(P + (int64_t)s * bb + o) = digit8(lo, hi, s);
}

// Base-16 planes in E4M3 (k_zgemm64): q = x 2^(56 - e) (|q| <= 2^56), then balanced digits from
// the least significant end, d_s in [-7, 8] for s >= 2, d_1 = what remains, in [-16, 16].
// Four adjacent elements (columns 4j .. 4j+3 of a row): one 32-bit store per plane.
__device__ __forceinline__ uint32_t e4m3_digit(int d) {
    return (uint32_t)(uint8_t)__nv_cvt_float_to_fp8((float)d, __NV_SATFINITE, __NV_E4M3);
}
__device__ __forceinline__ void put_digits4(const long long (&q0)[4], uint8_t *P, int64_t o, int64_t bb) {
    long long q[4] = {q0[0], q0[1], q0[2], q0[3]};
#pragma unroll
    for (int s = Z16_PLANES - 1; s >= 1; --s) {
        uint32_t w = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            int r = (int)(q[u] & 15);
            if (r > 8) r -= 16;
            q[u] = (q[u] - r) >> 4;
            w |= e4m3_digit(r) << (8 * u);
        }
        *reinterpret_cast<uint32_t *>(P + (int64_t)s * bb + o) = w;
    }
    uint32_t w = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) w |= e4m3_digit((int)q[u]) << (8 * u);
    *reinterpret_cast<uint32_t *>(P + o) = w;
}

// The planes of one b x b matrix at T (column-major; row-major when transpose) with digit
// exponent e into the slot at P (14 b^2 bytes, each plane row-major, K-major for the MMA).
// Blocks of 32 rows x 64 columns go through shared memory; a warp then writes whole 128-byte
// lines of 4 rows (FP16), or 32-byte sectors of 16 (E4M3).  Bound by the bytes (8 read, 14
// written an element) with the byte-permute digits; digit by digit with shifts and conversions
// the arithmetic took longer than the bytes (142 us for 16.3 tiles of 1024 on average).
template <bool E4M3>
__device__ __forceinline__ void planes_of_tile(const double *T, int b, bool transpose, int e, uint8_t *P) {
    __shared__ double S[64][33];
    const int nbr = b / 32, nbc = b / 64;
    const int64_t bb = (int64_t)b * b;
    for (int blk = blockIdx.x; blk < nbr * nbc; blk += gridDim.x) {
        const int r0 = (blk % nbr) * 32, c0 = (blk / nbr) * 64;
        __syncthreads();
        if (!transpose) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int idx = threadIdx.x + 256 * i, r = idx & 31, c = idx >> 5;
                S[c][r] = T[(int64_t)(c0 + c) * b + r0 + r];
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int idx = threadIdx.x + 256 * i, c = idx & 63, r = idx >> 6;
                S[c][r] = T[(int64_t)(r0 + r) * b + c0 + c];
            }
        }
        __syncthreads();
        if constexpr (!E4M3) {
            const int c = ((threadIdx.x >> 2) & 7) * 8, r = (threadIdx.x & 3) + 4 * (threadIdx.x >> 5);
            long long q[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) q[u] = fixed56(S[c + u][r], e);
            put_planes8(q, reinterpret_cast<__half *>(P), plane_at(b, r0 + r, c0 + c), bb);
        } else {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = (threadIdx.x & 7) * 4 + 32 * h, r = threadIdx.x >> 3;
                long long q[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) q[u] = fixed56(S[c + u][r], e);
                put_digits4(q, P, (int64_t)(r0 + r) * b + c0 + c, bb);
            }
        }
    }
}

// exps[t] = smallest e with amax[t] <= 2^e (Z_ZERO_EXP for a zero tile, whose digits are zero with any
// exponent); planes of tile t at pool + 14 t b^2.  The values come from tile t of W, or
// (alt != nullptr) from the blockIdx.y-th tile of the contiguous buffer alt.
template <bool E4M3>
__global__ void __launch_bounds__(256)
k_digits(const double *W, int b, const int *tiles, const double *amax, uint8_t *pool, int *exps, const double *alt) {
    const int t = tiles[blockIdx.y];
    const int64_t bb = (int64_t)b * b;
    const int e = z_digit_exp(amax[t]);
    if (blockIdx.x == 0 && threadIdx.x == 0) exps[t] = e;
    planes_of_tile<E4M3>(alt ? alt + (int64_t)blockIdx.y * bb : W + (int64_t)t * bb, b, false, e == Z_ZERO_EXP ? 0 : e,
                         pool + (int64_t)t * Z_SLOT * bb);
}

// --------------------------------------------------------------------- update kernel
// Work items: one 128 x ZBN block (bm, bn) of one output tile.  The kernel is persistent:
// CTA c takes items c, c + gridDim.x, ...; every role walks the same item sequence.

// In-core form: item i is items[i]; its sources are the consecutive digit slots
// it.xoff + n and it.yoff + n.
struct ZArgs {
    const uint8_t *pool;
    const ZItem *items;
    int nitems;
    const int *exps;
    int k, b;
    int *err;
    int assign;         // 0: C -= sum X Y^T;  1: C = sum X Y^T;  2: C = its counterpart in `add` + sum X Y^T
    const ZItem *add;   // assign 2: items whose C holds the summand
    double *amax;       // not null: largest |C| of the results of item it goes to amax[it.ct] (ct >= 0)
    int tri;            // 1: the Y tiles are lower triangular (row j is zero beyond column j)
    unsigned long long limit_ns;    // bound of each pipeline wait
    int stall;                      // test hook: wait first on a barrier nothing arrives at
    __device__ int count() const { return nitems; }
    __device__ bool tile(int i, ZItem &it) const {
        it = items[i];
        return true;
    }
    __device__ int xsrc(const ZItem &it, int n) const { return it.xoff + n; }
    __device__ int ysrc(const ZItem &it, int n) const { return it.yoff + n; }
    __device__ const double *base(const ZItem &it, int i) const { return assign == 2 ? add[i].C : it.C; }
    __device__ double *amax_of(const ZItem &it) const { return amax && it.ct >= 0 ? amax + it.ct : nullptr; }
};

// Out-of-core form: up to ZG_MAX output tiles of one tile column, whose sources sit in
// arbitrary cache slots; the slot lists travel in the launch parameters.  Item i of the
// ntiles x (b/ZBM) x (b/ZBN) blocks; blocks entirely above the diagonal of a `lower` tile
// carry no work.
struct ZGroupArgs {
    const uint8_t *pool;
    double *C[ZG_MAX];
    uint16_t xs[ZG_MAX][ZK_MAX];   // X_n of tile g: digit slot xs[g][n]
    uint16_t ys[ZK_MAX];           // Y_n (shared by the group): digit slot ys[n]
    const int *exps;
    int k, b, ntiles;
    int *err;
    int assign;
    int tri;
    uint32_t lower;                // bit g: tile g is a diagonal tile
    unsigned long long limit_ns;
    int stall;
    __device__ int count() const { return ntiles * (b / ZBM) * (b / ZBN); }
    __device__ bool tile(int i, ZItem &it) const {
        const int nbm = b / ZBM, per = nbm * (b / ZBN);
        const int g = i / per, r = i % per;
        it.C = C[g];
        it.xoff = g;
        it.yoff = 0;
        it.bm = (uint16_t)(r % nbm);
        it.bn = (uint16_t)(r / nbm);
        return !(((lower >> g) & 1u) && it.bm * ZBM + ZBM - 1 < it.bn * ZBN);
    }
    __device__ int xsrc(const ZItem &it, int n) const { return xs[it.xoff][n]; }
    __device__ int ysrc(const ZItem &, int n) const { return ys[n]; }
    __device__ const double *base(const ZItem &it, int) const { return it.C; }
    __device__ double *amax_of(const ZItem &) const { return nullptr; }
};

// Stages of ZKE elements of K that item `it` multiplies per source: all of them, or with a lower
// triangular Y only those up to the last column of Y's rows (the rest multiplies zeros).  This is
// what makes a TRSM product cost half an update's.
template <class Args>
__device__ __forceinline__ int z_kblocks(const Args &a, const ZItem &it) {
    const int all = a.b / ZKE;
    const int need = (it.bn * ZBN + ZBN - 1) / ZKE + 1;
    return a.tri && need < all ? need : all;
}

// Persistent update kernel: C -= sum_{n<k} X_n Y_n^T for 128 x ZBN output blocks, X_n the
// tiles (m, n) and Y_n the tiles (k, n), through their first P digit planes and the pairs
// s + t < P (launch_form below lists which P serves which output precision).
//   warp 0  copies: per source and 32 elements of K one stage, the P X planes of the
//           block's 128 rows and the P Y planes of its 32 columns;
//   warp 1  MMA issuer: per stage and X plane s, one tcgen05.mma per 16 elements of K with
//           N = ZBN (P - s) multiplies it by all its partners Y_0 .. Y_{P-1-s} at once; column
//           block t lands on accumulator group s + t, so the grouping by weight comes from the
//           TMEM address.  Plane 0 covers all groups and starts them at the head of a flush
//           period; elsewhere the long planes come last, so that their MMAs run while the thread
//           waits for the next stage;
//   warps 2-9 drain: every 128 elements of K the P group sums leave TMEM (exact FP32 integers)
//           and are added, shifted to the largest source's scale, to two int64 sums per element
//           that run over all sources of the item; FP64 arithmetic happens once per item.  (One
//           FP64 multiply-add per sum and source cost the FP64 pipe 5400 cycles at once, which
//           the MMAs then waited for: 10 % of the time at tile 1024, 40 % at tile 256.)
// The accumulators are double-buffered in TMEM (2 x P x ZBN = 448 columns), so a drain overlaps
// the next 128 elements' MMAs, and the item stream never stops between items (no per-item
// prologue).
// What bounds it: the tensor pipe.  Per 128 elements of K the 8 x 7 MMAs of P = 7 take
// 8 (112 + 96 + 80 + 64 + 48 + 2 x 41) = 3856 cycles for 128 x 32 outputs (an MMA takes
// max(41, N / 2) cycles).  Measured 4990 with boxes of 64-byte rows, of which 750 waited for a stage's
// copies (56 bytes a clock and SM, a row a clock); 4700 with bulk copies of the blocked planes, 450 of
// them waiting for stages and 270 for accumulators at the ends of items.  All P = 7 products of an FP64
// factorization of order 32768, tile 1024: 212 -> 197 ms (its updates alone took 346 ms with base 16
// in E4M3: 105 pairs, 128 x 16 items).  64 columns in two buffers do not fit TMEM.
//
// Failure handling: every pipeline wait gives up after args.limit_ns (or when another role
// set the abort flag), and the CTA then sets *err and stops issuing.  Before the TMEM is
// released and the CTA exits, the MMA issuer waits for all of its issued MMAs and the
// producer for all of its issued copies; those waits ignore the abort flag (the operations
// depend on nothing outside the CTA, so they end) and are bounded by ZDRAIN_NS.
template <int P, class Args>
__global__ void __maxnreg__(168)   // 320 threads: 3 warps on some SMSP x 32 x 168 <= 16K registers
k_zgemm(const __grid_constant__ Args args) {
    static_assert(P <= ZS && 2 * P * ZBN <= 512, "two accumulator buffers fit TMEM");
    extern __shared__ __align__(1024) uint8_t zsmem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(zsmem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + ZST * ZSTAGE);
    uint64_t *empty = full + ZST;
    uint64_t *accf = empty + ZST;                     // [2]
    uint64_t *acce = accf + 2;                        // [2]
    uint64_t *done = acce + 2;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(done + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_holder + 1);
    volatile int *never = abort_flag + 1;             // nothing sets it: waits that must not be cut short
    const unsigned long long lim = args.limit_ns;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = args.k, b = args.b;
    const int nitems = args.count();
    if ((int)blockIdx.x >= nitems) return;             // whole CTA, before any barrier
    if (threadIdx.x == 0) {
        for (int s = 0; s < ZST; ++s) {
            z_init(full + s, 1);
            z_init(empty + s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            z_init(accf + a, 1);
            z_init(acce + a, ZDRAIN);
        }
        z_init(done, 1);
        *abort_flag = 0;
        *never = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(z_smem(tmem_holder)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_holder;

    if (warp == 0) {
        // --------------------------------------------------------------- producer (bulk copies)
        int st = 0, ph = 1, issued = 0;             // empty slots: phase 1 passes
        const int64_t plane = 2 * (int64_t)b * b, slot = ZS * plane;
        bool ok = true;
        for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
            ZItem it;
            if (!args.tile(item, it)) continue;
            const int kblocks = z_kblocks(args, it);
            for (int n = 0; n < k && ok; ++n) {
                const uint8_t *x = args.pool + args.xsrc(it, n) * slot + it.bm * ZX_BYTES;
                const uint8_t *y = args.pool + args.ysrc(it, n) * slot + it.bn * ZY_BYTES;
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!z_wait_all(empty + st, ph, abort_flag, lim)) { ok = false; break; }
                    uint8_t *xs = smem + st * ZSTAGE, *ys = xs + ZS * ZX_BYTES;
                    z_expect_w(full + st, P * (ZX_BYTES + ZY_BYTES));
#pragma unroll
                    for (int s = 0; s < P; ++s) {
                        z_bulk_w(xs + s * ZX_BYTES, x + s * plane, ZX_BYTES, full + st);
                        z_bulk_w(ys + s * ZY_BYTES, y + s * plane, ZY_BYTES, full + st);
                    }
                    x += (int64_t)b * ZKB;
                    y += (int64_t)b * ZKB;
                    ++issued;
                    if (++st == ZST) { st = 0; ph ^= 1; }
                }
            }
        }
        if (!ok && lane == 0) {
            *abort_flag = 1;
            atomicExch(args.err, 1);
        }
        // Every copy lands before the shared memory goes away, whichever role gave up and
        // whenever: only the last ZST stages can still be in flight (each earlier one was
        // consumed before it was refilled), and each is the latest phase of its full barrier.
        // Without an abort they end as soon as those copies land.
        for (int q = issued - ZST < 0 ? 0 : issued - ZST; q < issued; ++q)
            if (!z_wait_all(full + q % ZST, (q / ZST) & 1, never, ZDRAIN_NS) && lane == 0) atomicExch(args.err, 3);
    } else if (warp == 1) {
        // --------------------------------------------------------------- MMA issuer
        // kind::f16, D F32, A/B F16, K-major, M = 128; N set per instruction
        const uint32_t idesc0 = (1u << 4) | ((uint32_t)(ZBM >> 4) << 24);
        // shared-memory descriptors advance by 2 per 32-byte K step (address field in
        // 16-byte units); stage index and phase run as counters (no division)
        const uint64_t desc0 = z_desc64(z_smem(smem));
        int st = 0, ph = 0, q = 0;                  // q: flush periods issued so far (all items)
        bool ok = true;
        // test hook: `done` completes only after the final commit below, so this wait runs
        // into the bound and takes the abort path
        if (args.stall && !z_wait_all(done, 0, abort_flag, lim)) ok = false;
        for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
            ZItem it;
            if (!args.tile(item, it)) continue;
            const int kblocks = z_kblocks(args, it);
            for (int n = 0; n < k && ok; ++n)
                for (int f0 = 0; f0 < kblocks && ok; f0 += ZFB, ++q) {
                    const int a = q & 1, f1 = f0 + ZFB < kblocks ? f0 + ZFB : kblocks;
                    if (!z_wait_all(acce + a, ((q >> 1) & 1) ^ 1, abort_flag, lim)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t dbase = tmem + (uint32_t)(a * P * ZBN);
                    for (int kb = f0; kb < f1; ++kb) {
                        if (!z_wait_all(full + st, ph, abort_flag, lim)) { ok = false; break; }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint64_t xd = desc0 + (uint64_t)((st * ZSTAGE) >> 4);
                        const uint64_t yd = xd + (uint64_t)((ZS * ZX_BYTES) >> 4);
                        if (kb == f0) {
                            z_mma2_h(dbase, xd, yd, idesc0 | ((uint32_t)((P * ZBN) >> 3) << 17), 0u);
#pragma unroll
                            for (int s = P - 1; s > 0; --s)
                                z_mma2_h(dbase + (uint32_t)(s * ZBN), xd + (uint64_t)((s * ZX_BYTES) >> 4), yd,
                                         idesc0 | ((uint32_t)(((P - s) * ZBN) >> 3) << 17), 1u);
                        } else {
#pragma unroll
                            for (int s = P - 1; s >= 0; --s)
                                z_mma2_h(dbase + (uint32_t)(s * ZBN), xd + (uint64_t)((s * ZX_BYTES) >> 4), yd,
                                         idesc0 | ((uint32_t)(((P - s) * ZBN) >> 3) << 17), 1u);
                        }
                        z_commit_w(empty + st);
                        if (++st == ZST) { st = 0; ph ^= 1; }
                    }
                    if (ok) z_commit_w(accf + a);
                }
        }
        if (!ok && lane == 0) {
            *abort_flag = 1;
            atomicExch(args.err, 1);
        }
        // every issued MMA completes before the TMEM is released and the CTA exits
        z_commit_w(done);
        if (!z_wait_all(done, 0, never, ZDRAIN_NS) && lane == 0) atomicExch(args.err, 3);
    } else {
        // --------------------------------------------------------------- drain + epilogue
        constexpr int COLS = ZBN / 2;                  // columns of a drain warp
        const int quarter = warp & 3, half = (warp - 2) >> 2;    // TMEM lanes 32 quarter.., columns 16 half..
        bool ok = true;
        int q = 0;
        for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
            ZItem it;
            if (!args.tile(item, it)) continue;
            const int kblocks = z_kblocks(args, it);
            // the largest scale of the item's sources: the unit of the sums (zero tiles cannot be it,
            // unless every source has one: then the sums are zero)
            int E0 = -(1 << 30);
            for (int n = lane; n < k; n += 32) E0 = max(E0, args.exps[args.xsrc(it, n)] + args.exps[args.ysrc(it, n)]);
            E0 = __reduce_max_sync(0xffffffffu, E0);
            // sum = 2^(E0 - 40) hi + 2^(E0 - 64) lo: a group g of a source of scale 2^E weighs
            // 2^(E - 16 - 8 g) = 2^(E0 - 64 + w), w = 48 - 8 g - (E0 - E); weights below one are
            // rounded to the unit 2^(E0 - 64), far below the truncation of the source of scale E0
            long long hi[COLS], lo[COLS];
#pragma unroll
            for (int j = 0; j < COLS; ++j) hi[j] = lo[j] = 0;
            for (int n = 0; n < k && ok; ++n) {
                const int w0 = 48 - E0 + args.exps[args.xsrc(it, n)] + args.exps[args.ysrc(it, n)];
                for (int f0 = 0; f0 < kblocks; f0 += ZFB, ++q) {
                    const int a = q & 1;
                    if (!z_wait(accf + a, (q >> 1) & 1, abort_flag, lim)) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t lanebase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * P * ZBN + half * COLS);
                    const auto add = [&](const float (&v)[16], int w) {
                        // group sums are exact integers: a 32-bit conversion (a 64-bit one would
                        // run on the FP64 pipe) and a 32 x 32 + 64 bit multiply-add
                        if (w >= 24) {
                            const int m = 1 << (w - 24);
#pragma unroll
                            for (int j = 0; j < COLS; ++j) hi[j] += (long long)__float2int_rn(v[j]) * m;
                        } else if (w >= 0) {
                            const int m = 1 << w;
#pragma unroll
                            for (int j = 0; j < COLS; ++j) lo[j] += (long long)__float2int_rn(v[j]) * m;
                        } else if (w > -28) {
                            const int sh = -w, r = 1 << (sh - 1);
#pragma unroll
                            for (int j = 0; j < COLS; ++j) lo[j] += (__float2int_rn(v[j]) + r) >> sh;
                        }
                    };
#pragma unroll
                    for (int g = 0; g < P; g += 2) {
                        float u[16], v[16];
                        if (g + 1 < P) z_ld16x2(lanebase + (uint32_t)(g * ZBN), lanebase + (uint32_t)((g + 1) * ZBN), u, v);
                        else z_ld16(lanebase + (uint32_t)(g * ZBN), u);
                        add(u, w0 - 8 * g);
                        if (g + 1 < P) add(v, w0 - 8 * (g + 1));
                    }
                    // the accumulator buffer is free for period q + 2 once every lane has read it
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) z_arrive(acce + a);
                }
            }
            if (!ok) break;
            const int row = it.bm * ZBM + quarter * 32 + lane;
            // all of C's values are requested before the first store, so the loads' latencies overlap
            // (one after another they cost 20000 cycles an item, which the MMAs then waited for)
            const int64_t o = (int64_t)(it.bn * ZBN + half * COLS) * b + row;
            const double *src = args.base(it, item) + o;
            double *c = it.C + o;
            double v[COLS];
#pragma unroll
            for (int j = 0; j < COLS; ++j) v[j] = args.assign == 1 ? 0.0 : src[(int64_t)j * b];
            unsigned long long m = 0;                  // sign-cleared bit patterns order like |x|
#pragma unroll
            for (int j = 0; j < COLS; ++j) {
                const double sum = fixed_sum(hi[j], lo[j], E0 - 64);
                const double out = args.assign == 1 ? sum : args.assign == 2 ? v[j] + sum : v[j] - sum;
                c[(int64_t)j * b] = out;
                m = max(m, (unsigned long long)__double_as_longlong(out) & 0x7FFFFFFFFFFFFFFFull);
            }
            if (double *am = args.amax_of(it)) {
#pragma unroll
                for (int w = 16; w > 0; w >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, w));
                if (lane == 0) atomicMax(reinterpret_cast<unsigned long long *>(am), m);
            }
        }
        if (!ok) {
            *abort_flag = 1;
            atomicExch(args.err, 1);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// Digit planes of one b x b matrix at src (column-major; row-major when transpose != 0)
// into slot dst of the pool, exponent from *amax.
template <bool E4M3>
__global__ void __launch_bounds__(256)
k_digits_src(const double *src, int b, int transpose, int dst, const double *amax, uint8_t *pool, int *exps) {
    const int e = z_digit_exp(*amax);
    if (blockIdx.x == 0 && threadIdx.x == 0) exps[dst] = e;
    planes_of_tile<E4M3>(src, b, transpose != 0, e == Z_ZERO_EXP ? 0 : e, pool + (int64_t)dst * Z_SLOT * b * b);
}

// max |src[e]| as the largest sign-cleared bit pattern (non-negative doubles order like their
// bit patterns; integer maxima keep this off the FP64 pipe)
__global__ void k_amax_ptr(const double *src, int64_t count, double *out) {
    unsigned long long m = 0;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        m = max(m, (unsigned long long)__double_as_longlong(src[e]) & 0x7FFFFFFFFFFFFFFFull);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned long long *>(out), m);
}

// zero the strictly upper part of a column-major b x b tile (a factored diagonal tile as L_kk)
__global__ void k_lower_only(double *T, int b) {
    const int64_t bb = (int64_t)b * b;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < bb; e += (int64_t)gridDim.x * blockDim.x)
        if (e % b < e / b) T[e] = 0.0;
}

__global__ void k_set_identity(double *T, int b) {
    const int64_t bb = (int64_t)b * b;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < bb; e += (int64_t)gridDim.x * blockDim.x)
        T[e] = (e % b == e / b) ? 1.0 : 0.0;
}

// CTAs of a conversion of ntiles tiles: one 32 x 64 block per pass, about eight CTAs per SM
static int digit_ctas(int ntiles, int b) {
    const int blocks = (b / 32) * (b / 64), want = tile_ctas(ntiles);
    return blocks < want ? blocks : want;
}
void launch_digits_src(const double *src, int b, int transpose, int dst, const double *amax, uint8_t *pool, int *exps,
                       cudaStream_t s, bool e4m3) {
    const int grid = digit_ctas(1, b);
    if (e4m3) k_digits_src<true><<<grid, 256, 0, s>>>(src, b, transpose, dst, amax, pool, exps);
    else k_digits_src<false><<<grid, 256, 0, s>>>(src, b, transpose, dst, amax, pool, exps);
}
void launch_amax_ptr(const double *src, int64_t count, double *out, cudaStream_t s) {
    const int64_t want = (count + 4095) / 4096;
    k_amax_ptr<<<want < 608 ? (int)want : 608, 256, 0, s>>>(src, count, out);
}
void launch_set_identity(double *T, int b, cudaStream_t s) { k_set_identity<<<64, 256, 0, s>>>(T, b); }

// ------------------------------------------------------------------------- host side
size_t zgemm_smem_bytes() { return (size_t)ZST * ZSTAGE + 1024 + 256; }

static int sm_count() {            // per device, cached
    static std::atomic<int> cache[64];
    int dev = 0;
    cudaGetDevice(&dev);
    std::atomic<int> &c = cache[dev & 63];
    int n = c.load(std::memory_order_relaxed);
    if (n <= 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 152;
        c.store(n, std::memory_order_relaxed);
    }
    return n;
}

void launch_digits(const double *W, int b, const int *tiles, int ntiles, const double *amax, uint8_t *pool, int *exps,
                   cudaStream_t s, bool e4m3, const double *alt) {
    if (ntiles <= 0) return;
    const dim3 grid(digit_ctas(ntiles, b), ntiles);
    if (e4m3) k_digits<true><<<grid, 256, 0, s>>>(W, b, tiles, amax, pool, exps, alt);
    else k_digits<false><<<grid, 256, 0, s>>>(W, b, tiles, amax, pool, exps, alt);
}
void launch_lower_only(double *T, int b, cudaStream_t s) { k_lower_only<<<64, 256, 0, s>>>(T, b); }
__global__ void k_add_tile(double *dst, const double *src, int64_t count) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        dst[e] += src[e];
}
void launch_add_tile(double *dst, const double *src, int b, cudaStream_t s) {
    k_add_tile<<<608, 256, 0, s>>>(dst, src, (int64_t)b * b);
}
// P planes of base 256 are worth 2P base-16 digits: they round an operand to 2^-(8P+1) of its
// scale, and the pairs they leave out stay below 2^-(8P) of the product's.
template <class Args>
static void launch_form(int planes, const Args &a, int nitems, cudaStream_t s) {
    static std::atomic<unsigned long long> attr{0};
    const size_t smem = zgemm_smem_bytes();
    if (attrs_pending(attr)) {
        cudaFuncSetAttribute(k_zgemm<7, Args>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(k_zgemm<5, Args>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(k_zgemm<4, Args>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(k_zgemm<3, Args>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(k_zgemm<2, Args>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        mark_attrs_set(attr);
    }
    const int grid = nitems < sm_count() ? nitems : sm_count();      // persistent: one CTA per SM
    if (planes == 10) k_zgemm<5, Args><<<grid, ZTHREADS, smem, s>>>(a);
    else if (planes == 7) k_zgemm<4, Args><<<grid, ZTHREADS, smem, s>>>(a);
    else if (planes == 6) k_zgemm<3, Args><<<grid, ZTHREADS, smem, s>>>(a);
    else if (planes == 4) k_zgemm<2, Args><<<grid, ZTHREADS, smem, s>>>(a);
    else k_zgemm<7, Args><<<grid, ZTHREADS, smem, s>>>(a);
}

void launch_zgemm(const uint8_t *pool, const ZItem *items, int nitems, const int *exps, int k,
                  int b, int *err, cudaStream_t s, int planes, int assign, int tri, unsigned long long limit_ns,
                  int stall, double *amax, const ZItem *add) {
    if (nitems <= 0 || k <= 0) return;
    const ZArgs a{pool, items, nitems, exps, k, b, err, assign, add, amax, tri, limit_ns ? limit_ns : ZLIMIT_NS, stall};
    launch_form(planes, a, nitems, s);
}

void launch_zgemm_group(const uint8_t *pool, const ZGroup &g, const int *exps, int b, int *err,
                        cudaStream_t s, int planes, int tri, unsigned long long limit_ns, int stall) {
    if (g.ntiles <= 0 || g.k <= 0) return;
    ZGroupArgs a;
    memset(&a, 0, sizeof a);
    a.pool = pool;
    for (int t = 0; t < g.ntiles; ++t) {
        a.C[t] = g.C[t];
        if (g.lower[t]) a.lower |= 1u << t;
        for (int n = 0; n < g.k; ++n) a.xs[t][n] = (uint16_t)g.xs[t][n];
    }
    for (int n = 0; n < g.k; ++n) a.ys[n] = (uint16_t)g.ys[n];
    a.exps = exps;
    a.k = g.k;
    a.b = b;
    a.ntiles = g.ntiles;
    a.err = err;
    a.assign = g.assign;
    a.tri = tri;
    a.limit_ns = limit_ns ? limit_ns : ZLIMIT_NS;
    a.stall = stall;
    launch_form(planes, a, g.ntiles * (b / ZBM) * (b / ZBN), s);
}

}  // namespace tc
