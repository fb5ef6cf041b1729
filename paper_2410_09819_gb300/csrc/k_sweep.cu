// Substitution sweeps as one kernel (Section III-D: forward L z = r, back L^T x = z), over 64-row
// blocks and groups of NQ right-hand sides; a group is a sweep of its own.
//
// Of a group's G CTAs, CTA c owns the row blocks c, c + G, c + 2G, ... (in the order of the sweep); all
// CTAs of the grid are resident (cooperative launch).  For its block a CTA streams the 64-wide
// panel of L that multiplies the solved part, as that part appears: `progress` counts a group's
// solved blocks, each CTA loads the next 64 x 64 block of L before it looks at the counter, and the
// block's own triangle waits in shared memory, scaled so that its solve needs no division on the
// chain.  Every CTA takes its blocks in sweep order and all CTAs are resident, so the block that a
// counter stands at always runs; every wait is bounded all the same and sets *err when it runs out.
//
// What bounds it: one right-hand side, the chain from block to block (counter and solution through
// L2, one 64 x 64 product, the 64-step triangle); many, the FP64 pipe (n^2 / 2 multiply-adds a
// sweep and column).  n = 32768, one column: 4.4 ms forward and 4.6 ms back, 9 us a block,
// where launches per tile with triangles of 256 rows in one CTA took 12.9 and 13.9 ms; n = 8192, 64
// columns: 4.0 and 4.2 ms, where they took 24.3 and 26.4 ms.
#include "tc_internal.h"
#include "zgemm_common.h"

#include <algorithm>

namespace tc {

constexpr unsigned long long SWEEP_LIMIT_NS = 4000000000ull;   // default bound of the wait for a block

__device__ __forceinline__ int sweep_progress(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// (one thread) the counter once it is above t; negative when another CTA gave up or the wait ran out
__device__ __forceinline__ int sweep_wait(const int *progress, int t, const int *err, unsigned long long limit_ns) {
    int v = sweep_progress(progress);
    if (v > t) return v;
    const uint64_t t0 = z_timer();
    while ((v = sweep_progress(progress)) <= t)
        if (*(const volatile int *)err || z_timer() - t0 > limit_ns) return -1;
    return v;
}

// element (0, 0) of the 64 x 64 block (i, j) of the factor, i >= j (leading dimension b)
__device__ __forceinline__ const double *sweep_block(const double *W, int b, int i, int j) {
    const int per = b >> 6, ti = i / per, tj = j / per;
    return W + tidx(ti, tj) * (int64_t)b * b + (int64_t)(j - tj * per) * 64 * b + (i - ti * per) * 64;
}

// a / d rounded once, from the reciprocal of d in two parts, hi = RN(1 / d) and lo = RN((1 - d hi) hi): RN(a hi + a lo)
// with a lo = part, where nothing on the way leaves the normal range; a division elsewhere.  A division
// takes a warp about eight FP64 instructions of 64 cycles, this two; the plain product a hi is rounded twice.
__device__ __forceinline__ double sweep_div(double a, double d, double hi, double part) {
    const uint64_t wa = (uint64_t)__double_as_longlong(a), wd = (uint64_t)__double_as_longlong(d);
    if (((uint32_t)(wa >> 52) & 2047) - 543u <= 960u && ((uint32_t)(wd >> 52) & 2047) - 543u <= 960u)
        return fma(a, hi, part);
    return wa << 1 == 0 ? a * hi : a / d;
}

// One warp solves a 64 x 64 triangle, given as the unit triangle M (forward: rows in order, M[j][c], c > j;
// backward: from the last row, M[j][c], c < j) and its diagonal M[j][j] with the reciprocals rhi + rlo; lane l
// holds elements l and l + 32.  A step of the chain is a shuffle and a multiply-add on the unit
// triangle's solution u; the elements themselves are u_j / M[j][j], of which the half solved first is
// divided while the chain runs through the other.
template <bool FWD>
__device__ __forceinline__ void sweep_tri(const double (*M)[65], const double *rhi, const double *rlo, double &u0, double &u1) {
    const int lane = threadIdx.x & 31;
    double &f = FWD ? u0 : u1, &g = FWD ? u1 : u0;     // solved first, solved second
    const int fi = FWD ? lane : lane + 32, gi = FWD ? lane + 32 : lane;
    if (FWD) {
#pragma unroll 8
        for (int j = 0; j < 32; ++j) {
            const double uj = __shfl_sync(0xffffffffu, u0, j);
            if (lane > j) u0 = fma(-uj, M[j][lane], u0);
            u1 = fma(-uj, M[j][lane + 32], u1);
        }
    } else {
#pragma unroll 8
        for (int j = 31; j >= 0; --j) {
            const double uj = __shfl_sync(0xffffffffu, u1, j);
            if (lane < j) u1 = fma(-uj, M[j + 32][lane + 32], u1);
            u0 = fma(-uj, M[j + 32][lane], u0);
        }
    }
    double part;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        if (c == 0) part = f * rlo[fi];
        if (c == 1) f = sweep_div(f, M[fi][fi], rhi[fi], part);
#pragma unroll
        for (int i = 8 * c; i < 8 * c + 8; ++i) {
            const int j = FWD ? i : 31 - i;
            const double uj = __shfl_sync(0xffffffffu, g, j);
            if (FWD ? lane > j : lane < j) g = fma(-uj, FWD ? M[j + 32][lane + 32] : M[j][lane], g);
        }
    }
    g = sweep_div(g, M[gi][gi], rhi[gi], g * rlo[gi]);
}

// In place on r (columns of nblk * 64 values, leading dimension ldr); group g = blockIdx.x % groups
// holds the columns g NQ ..  Step s of the sweep solves block s (forward) or nblk - 1 - s.
template <bool FWD, int NQ>
__global__ void __launch_bounds__(256, 2)
k_sweep(const double *__restrict__ W, int b, int nblk, double *r, int64_t ldr, int nrhs, int groups, int *progress,
        int *err, unsigned long long limit_ns, int stall) {
    // forward M[j][c] = l_cj / l_jj (c > j): u_j = z_j l_jj travels, z = u / l_jj at the end;
    // backward M[j][c] = l_jc / l_jj (c < j), likewise
    __shared__ double M[64][65], rhi[64], rlo[64];
    __shared__ __align__(16) double red[4 * NQ][64], xs[64][NQ];
    __shared__ int known, stop;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rr = tid & 63, part = tid >> 6;
    const int g = (int)blockIdx.x % groups, per = (int)gridDim.x / groups;
    const int nq = min(NQ, nrhs - g * NQ);
    double *rg = r + (int64_t)g * NQ * ldr;
    progress += g;
    for (int s = (int)blockIdx.x / groups; s < nblk; s += per) {
        const int i = FWD ? s : nblk - 1 - s;
        const double *Dg = sweep_block(W, b, i, i);
        __syncthreads();                               // the previous block's triangle is solved
        for (int idx = tid; idx < 4096; idx += 256) {
            const int rw = idx & 63, c = idx >> 6;
            if (rw >= c) {
                const double v = Dg[(int64_t)c * b + rw];
                if (FWD) M[c][rw] = v;
                else M[rw][c] = v;
            }
        }
        if (tid == 0) known = stop = 0;
        __syncthreads();
        if (tid < 64) {
            const double d = M[tid][tid], hi = 1.0 / d;
            rhi[tid] = hi;
            rlo[tid] = fma(-d, hi, 1.0) * hi;
        }
        __syncthreads();
        // rows p and 62 - p (backward 63 - p and p + 1) of the triangle have 64 elements together, row 31 (32) 32
        for (int p = warp; p < 32; p += 8)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q = lane + 32 * h, first = 63 - p;         // elements of the longer row
                if (p == 31 && h) break;
                const int k = q < first ? q : q - first;
                const int row = FWD ? (q < first ? p : 62 - p) : (q < first ? 63 - p : p + 1), col = FWD ? row + 1 + k : k;
                const double v = M[row][col];
                M[row][col] = sweep_div(v, M[row][row], rhi[row], v * rlo[row]);
            }
        // sum over the solved blocks t = 0 .. s - 1 (in sweep order).  Forward: thread (rr, part)
        // takes row rr and 16 columns of L; backward: warp w the columns 8w .. 8w + 7 of block column
        // i, a lane two adjacent rows of the solved block
        constexpr int NA = FWD ? (NQ == 1 ? 4 : NQ) : 8 * NQ;
        double acc[NA];
#pragma unroll
        for (int q = 0; q < NA; ++q) acc[q] = 0.0;
        double u0 = 0.0, u1 = 0.0;                     // a warp per right-hand side: its rows of r
        double *x = rg + (warp < nq ? warp : 0) * ldr + (int64_t)i * 64;
        if (warp < nq) {
            u0 = __ldcg(x + lane);
            u1 = __ldcg(x + lane + 32);
        }
        int have = 0;
        if (stall && s == 0 && tid == 0 && sweep_wait(progress, 0, err, limit_ns) < 0) stop = 1;     // test hook
        for (int t = 0; t < s; ++t) {
            const int j = FWD ? t : nblk - 1 - t;
            double l[16];
            if (FWD) {
                const double *B = sweep_block(W, b, i, j) + rr + (int64_t)(16 * part) * b;
#pragma unroll
                for (int q = 0; q < 16; ++q) l[q] = B[(int64_t)q * b];
            } else {
                const double2 *B = reinterpret_cast<const double2 *>(sweep_block(W, b, j, i) + (int64_t)(8 * warp) * b) + lane;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const double2 v = B[(int64_t)q * (b >> 1)];
                    l[2 * q] = v.x;
                    l[2 * q + 1] = v.y;
                }
            }
            __syncthreads();                           // xs of the previous block is read
            if (t >= have) {
                if (tid == 0) {
                    known = sweep_wait(progress, t, err, limit_ns);
                    if (known < 0) stop = 1;
                }
                __syncthreads();
                have = known;
                if (stop) break;
            }
            if (tid < 64 * NQ) xs[tid & 63][tid >> 6] = (tid >> 6) < nq ? __ldcg(rg + (tid >> 6) * ldr + (int64_t)j * 64 + (tid & 63)) : 0.0;
            __syncthreads();
            if (FWD) {
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    if constexpr (NQ == 1) {
                        acc[q & 3] = fma(l[q], xs[16 * part + q][0], acc[q & 3]);
                    } else {
#pragma unroll
                        for (int c = 0; c < NQ; ++c) acc[c] = fma(l[q], xs[16 * part + q][c], acc[c]);
                    }
                }
            } else {
#pragma unroll
                for (int c = 0; c < NQ; ++c) {
                    const double x0 = xs[2 * lane][c], x1 = xs[2 * lane + 1][c];
#pragma unroll
                    for (int q = 0; q < 8; ++q) acc[q * NQ + c] = fma(l[2 * q + 1], x1, fma(l[2 * q], x0, acc[q * NQ + c]));
                }
            }
        }
        __syncthreads();
        if (stop) {
            if (tid == 0) atomicExch(err, 1);
            return;
        }
        if (FWD) {
            if constexpr (NQ == 1) {
                red[part][rr] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
            } else {
#pragma unroll
                for (int c = 0; c < NQ; ++c) red[c * 4 + part][rr] = acc[c];
            }
        } else {
            // sums over the lanes: in every step a lane hands on the half of its sums that the other
            // lane keeps (9 additions a lane instead of 40 for one column, 31 instead of 160 for four,
            // and an addition holds its SM quarter for 64 cycles)
#pragma unroll
            for (int o = 16, n = 4 * NQ; o > 0; o >>= 1, n >>= 1) {
                const bool up = lane & o;
#pragma unroll
                for (int q = 0; q < 4 * NQ; ++q)
                    if (q < n) {
                        const double send = up ? acc[q] : acc[q + n], keep = up ? acc[q + n] : acc[q];
                        acc[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                if (n == 0) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
            }
            constexpr int LANES = 32 / (8 * NQ);
            const int q = lane / LANES;
            if (lane % LANES == 0) red[(q % NQ) * 4][8 * warp + q / NQ] = acc[0];
        }
        __syncthreads();
        if (warp < nq) {
            const double(*rd)[64] = red + 4 * warp;
            if (FWD) {
                u0 -= (rd[0][lane] + rd[1][lane]) + (rd[2][lane] + rd[3][lane]);
                u1 -= (rd[0][lane + 32] + rd[1][lane + 32]) + (rd[2][lane + 32] + rd[3][lane + 32]);
            } else {
                u0 -= rd[0][lane];
                u1 -= rd[0][lane + 32];
            }
            sweep_tri<FWD>(M, rhi, rlo, u0, u1);
            __stcg(x + lane, u0);
            __stcg(x + lane + 32, u1);
        }
        // (the release below covers the stores that the barrier orders before it)
        if constexpr (NQ == 1) __syncwarp();
        else __syncthreads();
        if (tid == 0) asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(progress), "r"(s + 1) : "memory");
    }
}

// Sweeps of nrhs columns; progress: SWEEP_GROUPS counters, cleared here.  Returns a cudaError_t.
template <bool FWD, int NQ>
static cudaError_t sweep_launch(const double *W, int b, int nblk, double *r, int64_t ldr, int nrhs, int *progress, int *err,
                                cudaStream_t s, unsigned long long limit_ns, int stall) {
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_sweep<FWD, NQ>, 256, 0);
    if (e != cudaSuccess) return e;
    // two CTAs per SM: more would share the SM's FP64 pipe with the block on the chain
    const int cap = sms * (occ < 2 ? occ : 2);
    if (cap < 1) return cudaErrorLaunchOutOfResources;
    for (int c0 = 0; c0 < nrhs;) {
        int groups = (nrhs - c0 + NQ - 1) / NQ;
        if (groups > SWEEP_GROUPS) groups = SWEEP_GROUPS;
        if (groups > cap) groups = cap;
        int per = cap / groups;
        if (per > nblk) per = nblk;
        int cols = nrhs - c0 < groups * NQ ? nrhs - c0 : groups * NQ;
        double *rc = r + (int64_t)c0 * ldr;
        if ((e = cudaMemsetAsync(progress, 0, groups * sizeof(int), s)) != cudaSuccess) return e;
        void *args[] = {(void *)&W, (void *)&b, (void *)&nblk, (void *)&rc, (void *)&ldr, (void *)&cols, (void *)&groups,
                        (void *)&progress, (void *)&err, (void *)&limit_ns, (void *)&stall};
        e = cudaLaunchCooperativeKernel((const void *)k_sweep<FWD, NQ>, dim3(groups * per), dim3(256), args, 0, s);
        if (e != cudaSuccess) return e;
        c0 += groups * NQ;
    }
    return cudaSuccess;
}
// Groups of four columns share a block of L in registers; up to three columns go as groups of one
// (their chains run side by side, and four-column groups would multiply padding).
int launch_sweep(const double *W, int b, int nblk, double *r, int64_t ldr, int nrhs, bool fwd, int *progress, int *err,
                 cudaStream_t s, unsigned long long limit_ns, int stall) {
    limit_ns = limit_ns ? std::max(limit_ns, GRID_WAIT_MIN_NS) : SWEEP_LIMIT_NS;
    if (nrhs < 4)
        return (int)(fwd ? sweep_launch<true, 1>(W, b, nblk, r, ldr, nrhs, progress, err, s, limit_ns, stall)
                         : sweep_launch<false, 1>(W, b, nblk, r, ldr, nrhs, progress, err, s, limit_ns, stall));
    return (int)(fwd ? sweep_launch<true, 4>(W, b, nblk, r, ldr, nrhs, progress, err, s, limit_ns, stall)
                     : sweep_launch<false, 4>(W, b, nblk, r, ldr, nrhs, progress, err, s, limit_ns, stall));
}

}  // namespace tc
