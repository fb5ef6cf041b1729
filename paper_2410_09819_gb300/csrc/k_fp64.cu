// FP64 kernels of the tile Cholesky: SYRK/GEMM updates (Algorithm 1's inner n-loop,
// Section III-A), the diagonal POTRF, the panel TRSM, and the substitution / residual
// kernels of the solve.  GB300's FP64 pipe issues about two DFMA per clock per SM
// (~1.05 TFLOP/s for the chip), so these kernels are DFMA-bound by a wide margin: the
// 64 x 64 register-blocked tile below keeps the pipe saturated from one CTA per SM.
#include "tc_internal.h"
#include "zgemm_common.h"

#define FIXED_FN __device__ __forceinline__
#include "fixed_exp.h"

#include <algorithm>
#include <cmath>

namespace tc {

// Right-hand-side kernels are compiled for 1, 4 and 16 columns: GB300 issues a DFMA for every
// unrolled column even when its predicate is off, and FP64 is its scarce pipe.
#define NQ_DISPATCH(nrhs, kern, grid, block, smem, stream, ...)                             \
    do {                                                                                  \
        if ((nrhs) <= 1) kern<1><<<(grid), (block), (smem), (stream)>>>(__VA_ARGS__);      \
        else if ((nrhs) <= 4) kern<4><<<(grid), (block), (smem), (stream)>>>(__VA_ARGS__); \
        else kern<16><<<(grid), (block), (smem), (stream)>>>(__VA_ARGS__);                \
    } while (0)


// acc (rows tx + 16 i, columns ty + 16 j of a 64 x 64 block) += X[:, k0:k1] Y[:, k0:k1]^T.
// X and Y point at the block's first row/column; column l of each is at l * ld.
__device__ __forceinline__ void dgemm_block(double (&acc)[4][4], const double *__restrict__ X,
                                            const double *__restrict__ Y, int ld, int k0, int k1,
                                            double (*Xs)[64], double (*Ys)[64]) {
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int k = k0; k < k1; k += 16) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int idx = tid + 256 * e, l = idx >> 6, r = idx & 63;
            const bool ok = (k + l) < k1;
            Xs[l][r] = ok ? X[(int64_t)(k + l) * ld + r] : 0.0;
            Ys[l][r] = ok ? Y[(int64_t)(k + l) * ld + r] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < 16; ++l) {
            double a[4], bb[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = Xs[l][tx + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) bb[j] = Ys[l][ty + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
        }
        __syncthreads();
    }
}

__device__ __forceinline__ bool failed(const int *status) {
    return status && *(volatile const int *)status != 0;
}

// ----------------------------------------------------------------------------- updates
__global__ void __launch_bounds__(256, 2)
k_dgemm_update(const DJob *__restrict__ jobs, const DItem *__restrict__ items, int ld,
               double *__restrict__ partials, const int *status) {
    __shared__ double Xs[16][64], Ys[16][64];
    const DItem it = items[blockIdx.x];
    const DJob jb = jobs[it.job];
    if (failed(status) || failed(jb.status)) return;
    const int i0 = it.bi * 64, j0 = it.bj * 64;
    double acc[4][4] = {};
    dgemm_block(acc, jb.X + i0, jb.Y + j0, ld, it.k0, it.k1, Xs, Ys);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    if (it.part < 0) {
        double *C = jb.C + (int64_t)j0 * ld + i0;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) C[(int64_t)(ty + 16 * j) * ld + tx + 16 * i] -= acc[i][j];
    } else {
        double *P = partials + (int64_t)it.part * 4096;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) P[(ty + 16 * j) * 64 + tx + 16 * i] = acc[i][j];
    }
}

__global__ void __launch_bounds__(256)
k_dgemm_reduce(const DRed *__restrict__ reds, int ld, const double *__restrict__ partials,
               const int *status) {
    if (failed(status)) return;
    const DRed r = reds[blockIdx.x];
    for (int e = 0; e < 16; ++e) {
        const int idx = threadIdx.x + 256 * e, rr = idx & 63, cc = idx >> 6;
        double s = 0.0;
        for (int p = 0; p < r.nparts; ++p) s += partials[(int64_t)(r.part0 + p) * 4096 + cc * 64 + rr];
        r.C[(int64_t)cc * ld + rr] -= s;
    }
}

// ------------------------------------------------------------------------------- POTRF
// Factor the 64 x 64 lower block at D in place (right-looking in shared memory).  A non-positive
// pivot records the 1-based global column in *status and stops.
//
// What bounds it: latency.  A dependent FP64 operation (a comparison too) takes 66 cycles, a division
// 440 and a square root 690, and a warp's FP64 instruction holds its SM quarter for 64 cycles whatever
// lanes are active.  So warps 0 and 1 run the chain, a thread per row with its element of the
// current column in a register: the pivot's root and its reciprocal in integer arithmetic
// (fixed_exp.h: the same correctly rounded values), one multiplication, one barrier, one
// multiply-add for the next column; warps 2 to 9 meanwhile take the previous step to the columns
// behind, through an element list in column order in which a finished column costs nothing.  Every
// element sees the same operations in the same order as in the plain loop.  A block took 94 us with a
// square root, a division and three barriers of 256 threads a step, 73 us with two barriers and
// FP64 comparisons on the chain, 52 us with the reciprocal's own Newton steps after the root and four
// warps on the rest, 38 us here (of a step's 1100 cycles the root and reciprocal take 490; a warp
// of its own for them, with named barriers, gains 5 %).
constexpr int POTRF_THREADS = 320;
__device__ __forceinline__ bool positive(double d) {       // d > 0 without the FP64 pipe
    const long long w = __double_as_longlong(d);
    return w > 0 && w <= 0x7FF0000000000000ll;
}
__device__ __forceinline__ void pivot_root(double d, double &sd, double &rp) {
    const int e = __double2hiint(d) >> 20;
    if (e > 100 && e < 1946) {
        fx::Num h, q;
        fx::sqrt_recip_rn(d, h, q);
        sd = fx::value(h);
        rp = fx::value(q);
    } else {
        sd = sqrt(d);
        rp = 1.0 / sd;
    }
}
__device__ __forceinline__ bool potrf64_body(double *D, int ld, int col0, int *status) {   // false: not positive
    __shared__ double S[64][65];                 // S[c][r], r >= c: L_rc once column c is done
    __shared__ double ls[2][64];                 // column j of L
    __shared__ int fail;
    __shared__ uint16_t tab[2080];               // elements (c << 8 | r), columns from the last to the first
    const int tid = threadIdx.x, warp = tid >> 5;
    for (int idx = tid; idx < 4096; idx += POTRF_THREADS) {
        const int r = idx & 63, c = idx >> 6;
        if (r >= c) {
            S[c][r] = __ldcg(D + (int64_t)c * ld + r);
            tab[(63 - c) * (64 - c) / 2 + r - c] = (uint16_t)(c << 8 | r);
        }
    }
    if (tid == 0) fail = 0;
    __syncthreads();
    if (warp < 2) {
        double z = S[0][tid], d = S[0][0];       // row tid of column j, and its pivot
        for (int j = 0; j < 64; ++j) {
            const int cur = j & 1;
            if (positive(d)) {
                double sd, rp;
                pivot_root(d, sd, rp);
                if (tid >= j) {
                    z = tid == j ? sd : z * rp;
                    ls[cur][tid] = z;
                    S[j][tid] = z;
                }
            } else if (tid == 0) {
                fail = j + 1;
            }
            __syncthreads();                     // column j is there, step j - 1 everywhere
            if (!positive(d)) break;
            if (j < 63) {
                const double l = ls[cur][j + 1];
                d = fma(-l, l, S[j + 1][j + 1]);
                if (tid > j) z = fma(-z, l, S[j + 1][tid]);
            }
        }
    } else {
        for (int j = 0; j < 64; ++j) {
            const int cur = j & 1;
            __syncthreads();
            if (fail) break;
            const int n = (62 - j) * (63 - j) / 2;        // elements of columns j + 2 ..
#pragma unroll 4
            for (int e = tid - 64; e < n; e += POTRF_THREADS - 64) {
                const int c = tab[e] >> 8, r = tab[e] & 63;
                S[c][r] = fma(-ls[cur][r], ls[cur][c], S[c][r]);
            }
        }
    }
    __syncthreads();
    if (fail) {
        if (tid == 0) atomicCAS(status, 0, col0 + fail);
        return false;
    }
    for (int idx = tid; idx < 4096; idx += POTRF_THREADS) {
        const int r = idx & 63, c = idx >> 6;
        if (r >= c) D[(int64_t)c * ld + r] = S[c][r];
    }
    return true;
}
__global__ void __launch_bounds__(POTRF_THREADS) k_potrf_block(double *D, int ld, int col0, int *status) {
    if (failed(status)) return;
    potrf64_body(D, ld, col0, status);
}

// Right-side solve of a strip of ROWS rows held in shared memory: X L^T = S in place, L the
// 64 x 64 lower block in Ls, rinv[j] = 1 / L[j][j].  Column j: X[r][j] = S[r][j] / L[j][j], then
// S[r][c] -= X[r][j] L[c][j] for c > j (threads: row tid % ROWS, columns step 256 / ROWS).
template <int ROWS>
__device__ __forceinline__ void strip_solve(double (*Ss)[65], double (*Ls)[65], const double *rinv) {
    const int tid = threadIdx.x, r = tid % ROWS, cg = tid / ROWS;
    constexpr int CS = 256 / ROWS;
    for (int j = 0; j < 64; ++j) {
        if (tid < ROWS) Ss[tid][j] *= rinv[j];
        __syncthreads();
        const double xrj = Ss[r][j];
        for (int c = j + 1 + cg; c < 64; c += CS) Ss[r][c] = fma(-xrj, Ls[c][j], Ss[r][c]);
        __syncthreads();
    }
}

// POTRF panel: rows below the factored 64-block within the diagonal tile, X L^T = C for
// PANEL_ROWS rows a CTA, one warp a row: lane l holds columns l and l + 32, x_j travels by shuffle,
// and no step needs a barrier.  Bound by the FP64 pipe (160 warp operations of 64 cycles a row, 10 us
// for 8 rows): a launch takes 17 us, where 16 rows with two block barriers a step took 28 us.
constexpr int PANEL_ROWS = 8;
__device__ __forceinline__ void panel_row(const double (*Ls)[65], const double *rinv, double &z0, double &z1) {
    const int lane = threadIdx.x & 31;
#pragma unroll 8
    for (int j = 0; j < 32; ++j) {
        const double x = __shfl_sync(0xffffffffu, z0, j) * rinv[j];
        if (lane > j) z0 = fma(-x, Ls[j][lane], z0);
        z1 = fma(-x, Ls[j][lane + 32], z1);
    }
#pragma unroll 8
    for (int j = 0; j < 32; ++j) {
        const double x = __shfl_sync(0xffffffffu, z1, j) * rinv[j + 32];
        if (lane > j) z1 = fma(-x, Ls[j + 32][lane + 32], z1);
    }
    z0 *= rinv[lane];
    z1 *= rinv[lane + 32];
}
__device__ __forceinline__ void panel_body(double *Pb, const double *L, int ld) {
    __shared__ double Ls[64][65], rinv[64];      // Ls[j][c] = l_cj, c >= j
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int idx = tid; idx < 4096; idx += 256) {
        const int c = idx & 63, j = idx >> 6;
        if (c >= j) Ls[j][c] = L[(int64_t)j * ld + c];
    }
    double z0 = Pb[(int64_t)lane * ld + warp], z1 = Pb[(int64_t)(lane + 32) * ld + warp];
    __syncthreads();
    if (tid < 64) rinv[tid] = 1.0 / Ls[tid][tid];
    __syncthreads();
    panel_row(Ls, rinv, z0, z1);
    Pb[(int64_t)lane * ld + warp] = z0;
    Pb[(int64_t)(lane + 32) * ld + warp] = z1;
}
__global__ void __launch_bounds__(256) k_trsm_rows(double *P, const double *L, int ld, const int *status) {
    if (failed(status)) return;
    panel_body(P + blockIdx.x * PANEL_ROWS, L, ld);
}

// One warp solves two rows x L^T = s in place (their chains interleave), Ls[j][c] = l_cj.
__device__ __forceinline__ void row_solve2(const double (*Ls)[65], double *s, double *t, const double *rinv) {
    const int lane = threadIdx.x & 31;
    double z0 = s[lane], z1 = s[lane + 32], y0 = t[lane], y1 = t[lane + 32];
#pragma unroll 8
    for (int j = 0; j < 32; ++j) {
        // the two rows' pivots in one multiplication: lanes 0 .. 15 hold one, 16 .. 31 the other
        const double zj = __shfl_sync(0xffffffffu, z0, j), yj = __shfl_sync(0xffffffffu, y0, j);
        const double p = (lane < 16 ? zj : yj) * rinv[j];
        const double xz = __shfl_sync(0xffffffffu, p, 0), xy = __shfl_sync(0xffffffffu, p, 16);
        const double l0 = Ls[j][lane], l1 = Ls[j][lane + 32];
        if (lane > j) {
            z0 = fma(-xz, l0, z0);
            y0 = fma(-xy, l0, y0);
        }
        z1 = fma(-xz, l1, z1);
        y1 = fma(-xy, l1, y1);
    }
#pragma unroll 8
    for (int j = 0; j < 32; ++j) {
        const double zj = __shfl_sync(0xffffffffu, z1, j), yj = __shfl_sync(0xffffffffu, y1, j);
        const double p = (lane < 16 ? zj : yj) * rinv[j + 32];
        const double xz = __shfl_sync(0xffffffffu, p, 0), xy = __shfl_sync(0xffffffffu, p, 16);
        const double l1 = Ls[j + 32][lane + 32];
        if (lane > j) {
            z1 = fma(-xz, l1, z1);
            y1 = fma(-xy, l1, y1);
        }
    }
    s[lane] = z0 * rinv[lane];
    s[lane + 32] = z1 * rinv[lane + 32];
    t[lane] = y0 * rinv[lane];
    t[lane + 32] = y1 * rinv[lane + 32];
}

// Column TRSM (Algorithm 1: A_mk = A_mk L_kk^{-T}): one CTA per 64-row strip of a tile,
// left-looking over the 64-column blocks of L_kk.
__global__ void __launch_bounds__(256, 2)
k_trsm_strips(const TStrip *__restrict__ strips, int ld, int b, const int *status) {
    if (failed(status) || failed(strips[blockIdx.x].status)) return;
    extern __shared__ double smem[];
    double(*Xs)[64] = reinterpret_cast<double(*)[64]>(smem);
    double(*Ys)[64] = reinterpret_cast<double(*)[64]>(smem + 16 * 64);
    double(*Ls)[65] = reinterpret_cast<double(*)[65]>(smem + 32 * 64);
    double(*Ss)[65] = reinterpret_cast<double(*)[65]>(smem + 32 * 64 + 64 * 65);
    double *rinv = smem + 32 * 64 + 2 * 64 * 65;
    const TStrip st = strips[blockIdx.x];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double *X = st.C + st.r0;
    for (int jb = 0; jb < b / 64; ++jb) {
        double acc[4][4] = {};
        dgemm_block(acc, X, st.L + jb * 64, ld, 0, jb * 64, Xs, Ys);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                Ss[tx + 16 * i][ty + 16 * j] = X[(int64_t)(jb * 64 + ty + 16 * j) * ld + tx + 16 * i] - acc[i][j];
        for (int idx = tid; idx < 4096; idx += 256) {
            const int r = idx & 63, c = idx >> 6;
            Ls[r][c] = (r >= c) ? st.L[(int64_t)(jb * 64 + c) * ld + jb * 64 + r] : 0.0;
        }
        __syncthreads();
        if (tid < 64) rinv[tid] = 1.0 / Ls[tid][tid];
        __syncthreads();
        strip_solve<64>(Ss, Ls, rinv);
        for (int idx = tid; idx < 4096; idx += 256) {
            const int r = idx & 63, c = idx >> 6;
            X[(int64_t)(jb * 64 + c) * ld + r] = Ss[r][c];
        }
        __syncthreads();
    }
}

// The same for 16-row strips, four times as many CTAs: for a column with too few 64-row strips to
// fill the SMs (each strip's b^2 / 2 multiply-adds a row run on one SM).  Products: a thread holds
// one row and four columns of the 16 x 64 block; triangles as in panel_body, a warp per row.
constexpr int SMALL_STRIP = 16;
__global__ void __launch_bounds__(256)
k_trsm_strips16(const TStrip *__restrict__ strips, int ld, int b, const int *status) {
    if (failed(status) || failed(strips[blockIdx.x].status)) return;
    __shared__ double M[64][65], rinv[64], buf[16 * SMALL_STRIP + 16 * 64];
    double(*Xs)[SMALL_STRIP] = reinterpret_cast<double(*)[SMALL_STRIP]>(buf);          // product operands ...
    double(*Ys)[64] = reinterpret_cast<double(*)[64]>(buf + 16 * SMALL_STRIP);
    double(*Ss)[65] = reinterpret_cast<double(*)[65]>(buf);                            // ... then the strip
    static_assert(SMALL_STRIP * 65 <= 16 * SMALL_STRIP + 16 * 64, "the strip fits the operands' place");
    const TStrip st = strips[blockIdx.x];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int tx = tid & 15, ty = tid >> 4;
    double *X = st.C + st.r0;
    for (int jb = 0; jb < b / 64; ++jb) {
        double acc[4] = {};
        const double *Lb = st.L + (int64_t)jb * 64;
        for (int k = 0; k < jb * 64; k += 16) {
            Xs[ty][tx] = X[(int64_t)(k + ty) * ld + tx];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int idx = tid + 256 * e;
                Ys[idx >> 6][idx & 63] = Lb[(int64_t)(k + (idx >> 6)) * ld + (idx & 63)];
            }
            __syncthreads();
#pragma unroll
            for (int l = 0; l < 16; ++l) {
                const double a = Xs[l][tx];
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[q] = fma(a, Ys[l][ty + 16 * q], acc[q]);
            }
            __syncthreads();
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) Ss[tx][ty + 16 * q] = X[(int64_t)(jb * 64 + ty + 16 * q) * ld + tx] - acc[q];
        for (int idx = tid; idx < 4096; idx += 256) {
            const int c = idx & 63, j = idx >> 6;
            if (c >= j) M[j][c] = Lb[(int64_t)(jb * 64 + j) * ld + c];
        }
        __syncthreads();
        if (tid < 64) rinv[tid] = 1.0 / M[tid][tid];
        __syncthreads();
        row_solve2(M, Ss[warp], Ss[warp + 8], rinv);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 4; ++q) X[(int64_t)(jb * 64 + ty + 16 * q) * ld + tx] = Ss[tx][ty + 16 * q];
        __syncthreads();
    }
}

// --------------------------------------------------------------------- tile bookkeeping
__device__ __forceinline__ double *diag_tile(double *W, int t, int b) {
    return W + ((int64_t)t * (t + 1) / 2 + t) * (int64_t)b * b;
}

// log|A| = 2 sum log L_ii over the n valid diagonal entries, fixed summation order.
__global__ void __launch_bounds__(1024) k_logdet(const double *W, int b, int64_t n, double *out) {
    __shared__ double red[1024];
    double s = 0.0;
    for (int64_t g = threadIdx.x; g < n; g += 1024) {
        const int t = (int)(g / b), r = (int)(g % b);
        const double *D = W + ((int64_t)t * (t + 1) / 2 + t) * (int64_t)b * b;
        s += log(D[(int64_t)r * b + r]);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 512; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = 2.0 * red[0];
}

// Padding of the last tile row: rows/columns >= n become those of the identity.
__global__ void k_fix_padding(double *W, int nt, int b, int64_t n) {
    const int j = blockIdx.y;                       // tile column in the last tile row
    const int i = nt - 1;
    const int nv = (int)(n - (int64_t)i * b);      // valid rows of the last tile row
    double *T = W + ((int64_t)i * (i + 1) / 2 + j) * (int64_t)b * b;
    const int64_t bb = (int64_t)b * b;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < bb; e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e % b), c = (int)(e / b);
        if (j < i) {
            if (r >= nv) T[e] = 0.0;
        } else if (r >= nv || c >= nv) {
            T[e] = (r == c) ? 1.0 : 0.0;
        }
    }
}

// Export clean-up: strictly upper parts of diagonal tiles and all padding become 0.
__global__ void k_zero_upper_diag(double *W, int nt, int b, int64_t n) {
    const int t = blockIdx.y;
    const int64_t bb = (int64_t)b * b;
    const int nv_last = (int)(n - (int64_t)(nt - 1) * b);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < bb; e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e % b), c = (int)(e / b);
        if (t < nt) {  // diagonal tile t
            double *D = W + ((int64_t)t * (t + 1) / 2 + t) * bb;
            const bool pad = (t == nt - 1) && (r >= nv_last || c >= nv_last);
            if (c > r || pad) D[e] = 0.0;
        } else {       // off-diagonal tile (nt-1, j) of the last tile row, j = t - nt
            const int j = t - nt, i = nt - 1;
            double *T = W + ((int64_t)i * (i + 1) / 2 + j) * bb;
            if (r >= nv_last) T[e] = 0.0;
        }
    }
}

// Sum the four per-part accumulators of each row in a fixed order and subtract them from
// R[q * ldr + g0 + r] (rows r of a 64-row chunk, RHS q < nrhs).
template <int NQ>
__device__ __forceinline__ void part_reduce_sub(double (*red)[17], const double (&acc)[NQ], int nrhs,
                                                double *R, int64_t ldr, int64_t g0) {
    const int tid = threadIdx.x, rr = tid & 63, part = tid >> 6;
    for (int p = 0; p < 4; ++p) {
        __syncthreads();
        if (part == p)
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nrhs) red[rr][q] = (p == 0) ? acc[q] : red[rr][q] + acc[q];
    }
    __syncthreads();
    for (int e = tid; e < 64 * nrhs; e += 256) {
        const int r = e % 64, q = e / 64;
        R[q * ldr + g0 + r] -= red[r][q];
    }
}

// -------------------------------------------------------------------------------- solves
// One warp solves the 64 x 64 triangle held in S (S[r][c] = L[r][c], r >= c) against the 64
// values in blk: forward (L x = blk) or backward (L^T x = blk).  Each lane owns rows lane and
// lane + 32; the solved value travels by shuffle, so the 64 steps need no block barrier, and
// the pivots' reciprocals are formed up front (x * (1/d): one extra rounding, off the chain).
__device__ __forceinline__ void warp_tri64(double (*S)[65], double *blk, bool forward) {
    const int lane = threadIdx.x & 31;
    double x0 = blk[lane], x1 = blk[lane + 32];
    const double r0 = 1.0 / S[lane][lane], r1 = 1.0 / S[lane + 32][lane + 32];
    if (forward) {
        for (int j = 0; j < 32; ++j) {
            if (lane == j) x0 *= r0;
            const double xj = __shfl_sync(0xffffffffu, x0, j);
            if (lane > j) x0 = fma(-S[lane][j], xj, x0);
            x1 = fma(-S[lane + 32][j], xj, x1);
        }
        for (int j = 0; j < 32; ++j) {
            if (lane == j) x1 *= r1;
            const double xj = __shfl_sync(0xffffffffu, x1, j);
            if (lane > j) x1 = fma(-S[lane + 32][32 + j], xj, x1);
        }
    } else {
        for (int j = 31; j >= 0; --j) {
            if (lane == j) x1 *= r1;
            const double xj = __shfl_sync(0xffffffffu, x1, j);
            if (lane < j) x1 = fma(-S[32 + j][lane + 32], xj, x1);
            x0 = fma(-S[32 + j][lane], xj, x0);
        }
        for (int j = 31; j >= 0; --j) {
            if (lane == j) x0 *= r0;
            const double xj = __shfl_sync(0xffffffffu, x0, j);
            if (lane < j) x0 = fma(-S[j][lane], xj, x0);
        }
    }
    blk[lane] = x0;
    blk[lane + 32] = x1;
}

// Forward substitution with one diagonal tile, one right-hand side r (in place): per 64-row
// block, the product with the solved part (256 threads, 4 partial sums per row, fixed order)
// and the warp solve of the diagonal block.
// T: the right-hand side's storage type (double, or float for the FP32 correction solves of a
// refined batched solve); the arithmetic is FP64 either way.
template <typename T>
__device__ __forceinline__ void fwd_diag_body(const double *L, int ld, int b, T *r) {
    __shared__ double red[4][64];
    __shared__ double blk[64];
    __shared__ double S[64][65];
    T *z = r;                            // solved in place (block barriers order the accesses)
    const int tid = threadIdx.x;
    const int rr = tid & 63, part = tid >> 6;
    for (int jb = 0; jb < b / 64; ++jb) {
        double acc = 0.0;
        for (int l = part; l < jb * 64; l += 4) acc = fma(L[(int64_t)l * ld + jb * 64 + rr], (double)z[l], acc);
        red[part][rr] = acc;
        for (int idx = tid; idx < 4096; idx += 256) {
            const int lr = idx & 63, lc = idx >> 6;
            S[lr][lc] = (lr >= lc) ? L[(int64_t)(jb * 64 + lc) * ld + jb * 64 + lr] : 0.0;
        }
        __syncthreads();
        if (tid < 64) blk[tid] = (double)z[jb * 64 + tid] - (red[0][tid] + red[1][tid] + red[2][tid] + red[3][tid]);
        __syncthreads();
        if (tid < 32) warp_tri64(S, blk, true);
        __syncthreads();
        if (tid < 64) z[jb * 64 + tid] = (T)blk[tid];
        __syncthreads();
    }
}

// Back substitution with one diagonal tile: L_jj^T x = z, one right-hand side (in place).
template <typename T>
__device__ __forceinline__ void bwd_diag_body(const double *L, int ld, int b, T *x) {
    __shared__ double S[64][65];
    __shared__ double red[4][64];
    __shared__ double blk[64];
    const int tid = threadIdx.x;
    const int rr = tid & 63, part = tid >> 6;
    for (int jb = b / 64 - 1; jb >= 0; --jb) {
        // acc[r] = sum_{l >= (jb+1)*64} L[l][jb*64 + r] x[l]: rows of the tile's column block,
        // read along l (column-major L: contiguous in l for a fixed column)
        double acc = 0.0;
        const double *Lc = L + (int64_t)(jb * 64 + rr) * ld;
        for (int l = (jb + 1) * 64 + part; l < b; l += 4) acc = fma(Lc[l], (double)x[l], acc);
        red[part][rr] = acc;
        for (int idx = tid; idx < 4096; idx += 256) {
            const int lr = idx & 63, lc = idx >> 6;
            S[lr][lc] = (lr >= lc) ? L[(int64_t)(jb * 64 + lc) * ld + jb * 64 + lr] : 0.0;
        }
        __syncthreads();
        if (tid < 64) blk[tid] = (double)x[jb * 64 + tid] - (red[0][tid] + red[1][tid] + red[2][tid] + red[3][tid]);
        __syncthreads();
        if (tid < 32) warp_tri64(S, blk, false);
        __syncthreads();
        if (tid < 64) x[jb * 64 + tid] = (T)blk[tid];
        __syncthreads();
    }
}

// R = B - A X (absmode 0) or R = |A| X (absmode 1, B unused) for the symmetric A held as
// lower tiles; rows and columns >= n (padding) contribute nothing and R's padding is 0.  A CTA takes
// 64 rows and one of the groups of NQ columns; the groups of the same rows are neighbours and
// find their tiles in L2.
// What bounds it: the FP64 pipe (n^2 multiply-adds a column).  Sixteen columns a CTA, a launch per
// sixteen, left SMs idle (128 CTAs at n = 8192) and each SM's pipe idle while its only CTA loaded.
// n = 8192, 64 columns: 12.6 ms that way, 8.6 ms with groups of eight side by side (the pipe's
// floor is 8.2 ms).
template <int NQ>
__global__ void __launch_bounds__(256)
k_symv_resid(const double *A, int nt, int b, int64_t n, const double *X, int64_t ldx,
             const double *B, int64_t ldb, double *R, int64_t ldr, int nrhs, int absmode) {
    __shared__ double xs[64][NQ];
    __shared__ double S[64][65];
    const int chunks = b / 64, groups = (nrhs + NQ - 1) / NQ;
    const int row = blockIdx.x / groups, q0 = (blockIdx.x % groups) * NQ;
    const int i = row / chunks, r0 = (row % chunks) * 64;
    X += q0 * ldx;
    B += q0 * ldb;
    R += q0 * ldr;
    nrhs = min(NQ, nrhs - q0);
    const int tid = threadIdx.x, rr = tid & 63, part = tid >> 6;
    const int64_t bb = (int64_t)b * b;
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    for (int j = 0; j < nt; ++j) {
        const bool lower = j <= i;
        const double *T = lower ? A + ((int64_t)i * (i + 1) / 2 + j) * bb : A + ((int64_t)j * (j + 1) / 2 + i) * bb;
        for (int c0 = 0; c0 < b; c0 += 64) {
            __syncthreads();
            for (int idx = tid; idx < 4096; idx += 256) {
                const int lo = idx & 63, hi = idx >> 6;
                double v;
                int64_t gr, gc;
                if (lower) {   // S[r][c] = A_ij[r0 + r][c0 + c], coalesced along r
                    v = T[(int64_t)(c0 + hi) * b + r0 + lo];
                    gr = (int64_t)i * b + r0 + lo; gc = (int64_t)j * b + c0 + hi;
                    if (gr >= n || gc >= n) v = 0.0;
                    S[lo][hi] = absmode ? fabs(v) : v;
                } else {       // S[r][c] = A_ji[c0 + c][r0 + r], coalesced along c
                    v = T[(int64_t)(r0 + hi) * b + c0 + lo];
                    gr = (int64_t)i * b + r0 + hi; gc = (int64_t)j * b + c0 + lo;
                    if (gr >= n || gc >= n) v = 0.0;
                    S[hi][lo] = absmode ? fabs(v) : v;
                }
            }
            for (int e = tid; e < 64 * nrhs; e += 256) {
                const int c = e % 64, q = e / 64;
                const int64_t g = (int64_t)j * b + c0 + c;
                xs[c][q] = (g < n) ? X[q * ldx + g] : 0.0;
            }
            __syncthreads();
            for (int c = part; c < 64; c += 4) {
                const double l = S[rr][c];
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (q < nrhs) acc[q] = fma(l, xs[c][q], acc[q]);
            }
        }
    }
    double(*red)[NQ + 1] = reinterpret_cast<double(*)[NQ + 1]>(&S[0][0]);
    for (int p = 0; p < 4; ++p) {
        __syncthreads();
        if (part == p)
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nrhs) red[rr][q] = (p == 0) ? acc[q] : red[rr][q] + acc[q];
    }
    __syncthreads();
    for (int e = tid; e < 64 * nrhs; e += 256) {
        const int r = e % 64, q = e / 64;
        const int64_t g = (int64_t)i * b + r0 + r;
        double out = 0.0;
        if (g < n) out = absmode ? red[r][q] : B[q * ldb + g] - red[r][q];
        R[q * ldr + g] = out;
    }
}

// One right-hand side: R = B - A x (ABS false) or R = |A| x (ABS true; x = ones when X is
// null), A symmetric and held as lower tiles (column-major, the diagonal tiles full).  One
// CTA per 64 rows [r0, r0 + 64) of tile row i; every element of its 64 x n row panel is
// loaded once, straight from global memory into registers, for one multiply-add.
//   * tiles A_ij, j <= i: columns of the stored tile.  Warp w takes the columns c = w (mod 8),
//     each lane two adjacent rows (one 16-byte load per column; a warp reads 512 contiguous
//     bytes), with two accumulators per row so that consecutive columns do not chain.
//   * tiles right of the diagonal, A_ij = A_ji^T (j > i): row r of A_ij is column r of the
//     stored A_ji, contiguous in memory.  Warp w takes the rows r0 + 8w ... r0 + 8w + 7, its
//     lanes two adjacent columns per 64, with x's pair loaded once for the eight rows.
// Partial sums meet in a fixed order (lanes by shuffle, warps in shared memory), so the
// result does not depend on scheduling.  Rows and columns >= n (padding) contribute nothing
// and R's padding is 0.  The multiply-adds, not the bytes, bound it: a GB300 SM retires two
// FP64 multiply-adds per clock, n^2 per call.
template <bool ABS>
__global__ void __launch_bounds__(256)
k_symv1(const double *__restrict__ A, int nt, int b, int64_t n, const double *__restrict__ X,
        const double *__restrict__ B, double *__restrict__ R) {
    __shared__ double red[8][64];
    __shared__ double tr[64];
    const int chunks = b / 64;
    const int i = blockIdx.x / chunks, r0 = (blockIdx.x % chunks) * 64;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t bb = (int64_t)b * b;
    // tiles left of and on the diagonal
    double a0 = 0.0, a1 = 0.0, e0 = 0.0, e1 = 0.0;
    for (int j = 0; j <= i; ++j) {
        const double *T = A + ((int64_t)i * (i + 1) / 2 + j) * bb + r0 + 2 * lane;
        const double *x = X ? X + (int64_t)j * b : nullptr;
        const int cmax = (int)min((int64_t)b, n - (int64_t)j * b);
        int c = warp;
#pragma unroll 2
        for (; c + 8 < cmax; c += 16) {
            const double2 v = __ldg(reinterpret_cast<const double2 *>(T + (int64_t)c * b));
            const double2 w = __ldg(reinterpret_cast<const double2 *>(T + (int64_t)(c + 8) * b));
            const double xv = x ? __ldg(x + c) : 1.0, xw = x ? __ldg(x + c + 8) : 1.0;
            a0 = fma(ABS ? fabs(v.x) : v.x, xv, a0);
            a1 = fma(ABS ? fabs(v.y) : v.y, xv, a1);
            e0 = fma(ABS ? fabs(w.x) : w.x, xw, e0);
            e1 = fma(ABS ? fabs(w.y) : w.y, xw, e1);
        }
        if (c < cmax) {
            const double2 v = __ldg(reinterpret_cast<const double2 *>(T + (int64_t)c * b));
            const double xv = x ? __ldg(x + c) : 1.0;
            a0 = fma(ABS ? fabs(v.x) : v.x, xv, a0);
            a1 = fma(ABS ? fabs(v.y) : v.y, xv, a1);
        }
    }
    red[warp][2 * lane] = a0 + e0;
    red[warp][2 * lane + 1] = a1 + e1;
    // tiles right of the diagonal, through the stored tiles (j, i)
    double acc[8];
#pragma unroll
    for (int p = 0; p < 8; ++p) acc[p] = 0.0;
    for (int j = i + 1; j < nt; ++j) {
        const double *T = A + ((int64_t)j * (j + 1) / 2 + i) * bb + (int64_t)(r0 + 8 * warp) * b + 2 * lane;
        const double *x = X ? X + (int64_t)j * b + 2 * lane : nullptr;
        const int cmax = (int)min((int64_t)b, n - (int64_t)j * b);
        for (int m = 0; m < b; m += 64) {
            double2 xv = x ? __ldg(reinterpret_cast<const double2 *>(x + m)) : make_double2(1.0, 1.0);
            const int c = m + 2 * lane;
            if (c >= cmax) xv.x = 0.0;
            if (c + 1 >= cmax) xv.y = 0.0;
            const bool lo = c < cmax, hi = c + 1 < cmax;
#pragma unroll
            for (int p = 0; p < 8; ++p) {
                double2 v = __ldg(reinterpret_cast<const double2 *>(T + (int64_t)p * b + m));
                if (!lo) v.x = 0.0;
                if (!hi) v.y = 0.0;
                acc[p] = fma(ABS ? fabs(v.x) : v.x, xv.x, acc[p]);
                acc[p] = fma(ABS ? fabs(v.y) : v.y, xv.y, acc[p]);
            }
        }
    }
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        double v = acc[p];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) tr[8 * warp + p] = v;
    }
    __syncthreads();
    if (threadIdx.x < 64) {
        const int r = threadIdx.x;
        double s = tr[r];
#pragma unroll
        for (int w = 0; w < 8; ++w) s += red[w][r];
        const int64_t g = (int64_t)i * b + r0 + r;
        double out = 0.0;
        if (g < n) out = ABS ? s : B[g] - s;
        R[g] = out;
    }
}

// out[c] = max_r |V[c*ld + r]|, r < n (out must start at 0; max of non-negative doubles is
// monotone in their bit patterns, so atomicMax on the bits is exact and order-free).
__global__ void k_colmax_abs(const double *V, int64_t ld, int64_t n, double *out) {
    const int c = blockIdx.y;
    double m = 0.0;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
        m = fmax(m, fabs(V[c * ld + r]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(reinterpret_cast<unsigned long long *>(out + c), (unsigned long long)__double_as_longlong(m));
}

__global__ void k_axpy_cols(double *X, int64_t ldx, const double *D, int64_t ldd, int64_t n) {
    const int c = blockIdx.y;
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
        X[c * ldx + r] += D[c * ldd + r];
}

__global__ void __launch_bounds__(1024) k_dot_self(const double *v, int64_t n, double *out) {
    __shared__ double red[1024];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += 1024) s = fma(v[i], v[i], s);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 512; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}


// Batched POTRF step: one CTA per matrix entry (same 64-block position in each).
__global__ void __launch_bounds__(POTRF_THREADS) k_potrf_blocks(const PEntry *__restrict__ e, int ld) {
    const PEntry E = e[blockIdx.x];
    if (failed(E.status)) return;
    potrf64_body(E.D, ld, E.col0, E.status);
}

// Batched POTRF panel: rows below each entry's factored 64-block (grid.y = entry).
__global__ void __launch_bounds__(256) k_trsm_rows_batched(const PEntry *__restrict__ e, int ld) {
    const PEntry E = e[blockIdx.y];
    if (failed(E.status) || (int)blockIdx.x * PANEL_ROWS >= E.rows) return;
    panel_body(E.D + 64 + blockIdx.x * PANEL_ROWS, E.D, ld);
}

void launch_potrf_blocks(const PEntry *e, int n, int ld, cudaStream_t s) {
    if (n > 0) k_potrf_blocks<<<n, POTRF_THREADS, 0, s>>>(e, ld);
}
void launch_trsm_rows_batched(const PEntry *e, int n, int max_rows, int ld, cudaStream_t s) {
    if (n > 0 && max_rows > 0) k_trsm_rows_batched<<<dim3(max_rows / PANEL_ROWS, n), 256, 0, s>>>(e, ld);
}


// POTRF trailing update: C -= P P^T with the 64 columns P below the factored block at D, on the
// 64 x 64 blocks of the lower part (diagonal ones whole), sixteen CTAs of 16 x 16 elements each.  The
// FP64 pipe bounds it (1.7 multiply-adds a clock and SM): one CTA a 64 x 64 block keeps its SM busy for
// 69 us, and the 15 x 16 / 2 of them below the first panel of a 1024 tile are fewer than the SMs, so
// every step took 69 us (35 us on average in blocks of 32 x 32, 27 us in these).  At tile 2048 the 84 us
// of a step are the pipe's.
constexpr int SYRK_B = 16, SYRK_THREADS = 64;
__device__ __forceinline__ void syrk_body(double *D, int ld) {
    __shared__ double X[64][SYRK_B], Y[64][SYRK_B];
    const int t = blockIdx.x >> 4, tid = threadIdx.x;
    int bi = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while (bi * (bi + 1) / 2 > t) --bi;
    while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
    const int bj = 4 * (t - bi * (bi + 1) / 2) + ((blockIdx.x >> 2) & 3);
    bi = 4 * bi + (blockIdx.x & 3);
    const double *P = D + 64;
    double *C = D + (int64_t)(64 + bj * SYRK_B) * ld + 64 + bi * SYRK_B;
    const int r = tid & 15, q = tid >> 4;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        X[q + 4 * k][r] = P[(int64_t)(q + 4 * k) * ld + bi * SYRK_B + r];
        Y[q + 4 * k][r] = P[(int64_t)(q + 4 * k) * ld + bj * SYRK_B + r];
    }
    // a row and four columns a thread
    double acc[4] = {};
    __syncthreads();
#pragma unroll 16
    for (int k = 0; k < 64; ++k) {
        const double a = X[k][r];
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] = fma(a, Y[k][q + 4 * c], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) C[(int64_t)(q + 4 * c) * ld + r] -= acc[c];
}
__global__ void __launch_bounds__(SYRK_THREADS) k_syrk_rows_batched(const PEntry *__restrict__ e, int ld) {
    const PEntry E = e[blockIdx.y];
    if (!failed(E.status)) syrk_body(E.D, ld);
}
__global__ void __launch_bounds__(SYRK_THREADS) k_syrk_rows(double *D, int ld, const int *status) {
    if (!failed(status)) syrk_body(D, ld);
}
void launch_syrk_rows_batched(const PEntry *e, int n, int rows, int ld, cudaStream_t s) {
    const int m = rows / 64;
    for (int i = 0; i < n && m > 0; i += 65535)
        k_syrk_rows_batched<<<dim3(8 * m * (m + 1), n - i < 65535 ? n - i : 65535), SYRK_THREADS, 0, s>>>(e + i, ld);
}
void launch_syrk_rows(double *D, int rows, int ld, const int *status, cudaStream_t s) {
    const int m = rows / 64;
    if (m > 0) k_syrk_rows<<<8 * m * (m + 1), SYRK_THREADS, 0, s>>>(D, ld, status);
}

// The whole POTRF of one tile as a cooperative kernel: CTA 0 factors the 64-blocks of the diagonal, the
// others solve the panels and update the trailing blocks, all with the operations and the order of
// the kernels above (the same bits).  What this is for: the chain.  A step's three launches took
// 38 + 17 + 27 us and the gaps between them at tile 1024 although only 16 of the update's blocks stand
// before the next pivot block.  Here those 16 come first, alone on their SMs, and the next 64-block is
// factored while the rest of the update runs; they take the whole CTA, an element a thread (a group of two
// warps needs 8 us for a block's multiply-adds, eight warps 2), and the panel's rows are loaded
// while their block is factored.  A step takes 61 us at tile 1024 (86 as launches), 58 at tile 512 (77),
// 112 at tile 2048 (143; the pipe's own 84).
//   * flags[0 ..]: block j is factored (-1: not positive, everyone leaves); [64 ..]: CTAs done with panel
//     j; [128 ..] and [192 ..]: updates of diagonal block j and of block column j through step j - 1.
//   * A 16 x 16 block belongs to one group of 64 threads for good, so its updates are in order without
//     flags; index e counts from the last block column, so what trails step j are the first
//     8 m (m + 1) indexes and a group takes its own from the top: diagonal block, its column, the rest.
//   * Data of other CTAs is read through L2 (ld.cg), and every wait is bounded: a wait that runs out
//     sets *err, and all CTAs leave.
constexpr int PT_GROUPS = POTRF_THREADS / 64, PT_FLAGS = 64;
constexpr size_t PT_SMEM = (size_t)PT_GROUPS * 2 * 64 * SYRK_B * sizeof(double);
constexpr unsigned long long PT_LIMIT_NS = 4000000000ull;
static_assert(PT_SMEM >= (64 * 65 + 64) * sizeof(double), "a panel's triangle fits the update's place");

// (one thread) waits until *p is at least want; negative when it turned negative or the wait ran out
__device__ __forceinline__ int pt_wait(const int *p, int want, int *err, unsigned long long limit_ns) {
    int v;
    const uint64_t t0 = z_timer();
    for (;;) {
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        if (v >= want || v < 0) return v;
        if (*(volatile int *)err) return -1;
        if (z_timer() - t0 > limit_ns) {
            atomicExch(err, ERR_POTRF_WAIT);
            return -1;
        }
    }
}
__device__ __forceinline__ void pt_add(int *p) {          // (one thread, after a barrier) releases the CTA's or group's stores
    __threadfence();
    atomicAdd(p, 1);
}
__device__ __forceinline__ void pt_group_sync(int grp) { asm volatile("bar.sync %0, 64;" ::"r"(grp + 1) : "memory"); }

__global__ void __launch_bounds__(POTRF_THREADS)
k_potrf_tile(double *D, int ld, int nb, int col0, int *status, int *flags, int *err, unsigned long long limit_ns,
             int stall) {
    extern __shared__ double pts[];
    __shared__ int ready, go, filled;    // a flag per wait of a step, so that its next write comes after a barrier
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int *factored = flags, *panels = flags + PT_FLAGS, *diag = flags + 2 * PT_FLAGS, *column = flags + 3 * PT_FLAGS;
    // a tile after a failure: nothing runs (a failure in this call comes after every CTA's first panel)
    if (tid == 0) go = !failed(status);
    __syncthreads();
    if (blockIdx.x == 0) {
        if (!go) {
            if (tid == 0) atomicExch(factored, -1);
            return;
        }
        for (int j = 0; j < nb; ++j) {
            if (j > 0 || stall) {                          // (block 0 has no updates: the test hook's wait runs out)
                if (tid == 0) go = pt_wait(diag + j, 16, err, limit_ns) > 0;
                __syncthreads();
                if (!go) return;
            }
            const bool ok = potrf64_body(D + (int64_t)j * 64 * ld + j * 64, ld, col0 + j * 64, status);
            __syncthreads();
            if (tid == 0) {
                __threadfence();
                atomicExch(factored + j, ok ? 1 : -1);
            }
            if (!ok) return;
        }
        return;
    }
    const int w = (int)blockIdx.x - 1, nw = (int)gridDim.x - 1, grp = tid >> 6, gt = tid & 63;
    for (int j = 0; j + 1 < nb; ++j) {
        const int m = nb - 1 - j;                          // block rows below
        const int g0 = w + nw * (warp >> 2);               // the panel: four adjacent rows to four warps, eight warps a CTA
        const bool mine = warp < 8 && g0 < 16 * m;
        double *const Pr = D + (int64_t)(j * 64 + lane) * ld + (j + 1) * 64 + (warp & 3);
        const int64_t half = (int64_t)32 * ld;
        double z0 = 0.0, z1 = 0.0;
        if (tid == 0) ready = j == 0 || pt_wait(column + j, 16 * (m + 1), err, limit_ns) > 0;
        __syncthreads();
        if (!ready) return;
        if (mine) {                                        // the first rows, while block j is factored
            z0 = __ldcg(Pr + 4 * g0);
            z1 = __ldcg(Pr + 4 * g0 + half);
        }
        if (tid == 0) go = pt_wait(factored + j, 1, err, limit_ns) > 0;
        __syncthreads();
        if (!go) return;
        if (w < 16 * m) {
            double(*Ls)[65] = reinterpret_cast<double(*)[65]>(pts), *rinv = pts + 64 * 65;
            const double *L = D + (int64_t)j * 64 * ld + j * 64;
#pragma unroll 4
            for (int idx = tid; idx < 4096; idx += POTRF_THREADS) {
                const int c = idx & 63, k = idx >> 6;
                if (c >= k) Ls[k][c] = __ldcg(L + (int64_t)k * ld + c);
            }
            __syncthreads();
            if (tid < 64) rinv[tid] = 1.0 / Ls[tid][tid];
            __syncthreads();
            if (mine)
                for (int g = g0; g < 16 * m; g += 2 * nw) {
                    if (g != g0) {
                        z0 = __ldcg(Pr + 4 * g);
                        z1 = __ldcg(Pr + 4 * g + half);
                    }
                    panel_row(Ls, rinv, z0, z1);
                    __stcg(Pr + 4 * g, z0);
                    __stcg(Pr + 4 * g + half, z1);
                }
        }
        __syncthreads();
        if (tid == 0) {
            pt_add(panels + j);
            filled = pt_wait(panels + j, nw, err, limit_ns) > 0;
        }
        __syncthreads();
        if (!filled) return;
        const int total = 8 * m * (m + 1), slots = PT_GROUPS * nw, slot = grp * nw + w;
        int e = slot < total ? slot + (total - 1 - slot) / slots * slots : -1;
        double(*X)[SYRK_B] = reinterpret_cast<double(*)[SYRK_B]>(pts + (size_t)grp * 2 * 64 * SYRK_B), (*Y)[SYRK_B] = X + 64;
        const int r = gt & 15, q = gt >> 4;
        const double *P = D + (int64_t)j * 64 * ld;
        // the blocks of the next diagonal block on the whole CTA, an element a thread
        for (int t = total - 16; t < total; ++t) {
            if (t % slots % nw != w) continue;
            const int bi = 4 * (j + 1) + (t & 3), bj = 4 * (j + 1) + ((t >> 2) & 3), col = tid >> 4;
            double(*XA)[SYRK_B] = reinterpret_cast<double(*)[SYRK_B]>(pts), (*YA)[SYRK_B] = XA + 64;
            const int64_t o = (int64_t)(bj * SYRK_B + col) * ld + bi * SYRK_B + r;
            double acc = 0.0, old = 0.0;
            if (tid < 256) {
                old = __ldcg(D + o);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    XA[col + 16 * k][r] = __ldcg(P + (int64_t)(col + 16 * k) * ld + bi * SYRK_B + r);
                    YA[col + 16 * k][r] = __ldcg(P + (int64_t)(col + 16 * k) * ld + bj * SYRK_B + r);
                }
            }
            __syncthreads();
            if (tid < 256) {
#pragma unroll 16
                for (int k = 0; k < 64; ++k) acc = fma(XA[k][r], YA[k][col], acc);
                __stcg(D + o, old - acc);
            }
            __syncthreads();
            if (tid == 0) {
                pt_add(diag + j + 1);
                pt_add(column + j + 1);
            }
        }
        if (e >= total - 16) e -= slots;
        const auto update = [&](int id) {
            const int t = id >> 4;
            int c = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
            while (c * (c + 1) / 2 > t) --c;
            while ((c + 1) * (c + 2) / 2 <= t) ++c;
            const int bi = 4 * (nb - 1 - (t - c * (c + 1) / 2)) + (id & 3), bj = 4 * (nb - 1 - c) + ((id >> 2) & 3);
            double *C = D + (int64_t)bj * SYRK_B * ld + bi * SYRK_B;
            pt_group_sync(grp);                            // the previous block's operands are used
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                X[q + 4 * k][r] = __ldcg(P + (int64_t)(q + 4 * k) * ld + bi * SYRK_B + r);
                Y[q + 4 * k][r] = __ldcg(P + (int64_t)(q + 4 * k) * ld + bj * SYRK_B + r);
            }
            double acc[4] = {}, old[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) old[u] = __ldcg(C + (int64_t)(q + 4 * u) * ld + r);
            pt_group_sync(grp);
#pragma unroll 16
            for (int k = 0; k < 64; ++k) {
                const double a = X[k][r];
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[u] = fma(a, Y[k][q + 4 * u], acc[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) __stcg(C + (int64_t)(q + 4 * u) * ld + r, old[u] - acc[u]);
            if (c == m - 1) {                              // block column j + 1
                pt_group_sync(grp);
                if (gt == 0) pt_add(column + j + 1);
            }
        };
        for (; e >= 0; e -= slots) update(e);
    }
}
size_t potrf_tile_flags() { return 4 * PT_FLAGS * sizeof(int); }
// A tile whose steps fit the flags, from two 64-blocks on; the grid is what the first update keeps busy.
bool potrf_tile_ok(int b) { return b >= 128 && b <= 64 * PT_FLAGS; }
int launch_potrf_tile(double *D, int b, int col0, int *status, int *flags, int *err, cudaStream_t s,
                      unsigned long long limit_ns, int stall) {
    static std::atomic<unsigned long long> attr{0};
    if (attrs_pending(attr)) {
        cudaFuncSetAttribute(k_potrf_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PT_SMEM);
        mark_attrs_set(attr);
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMemsetAsync(flags, 0, potrf_tile_flags(), s);
    if (e != cudaSuccess) return (int)e;
    int nb = b / 64, grid = 1 + 8 * nb * (nb - 1);
    if (grid > sms) grid = sms;
    limit_ns = limit_ns ? std::max(limit_ns, GRID_WAIT_MIN_NS) : PT_LIMIT_NS;
    void *args[] = {(void *)&D, (void *)&b, (void *)&nb, (void *)&col0, (void *)&status, (void *)&flags, (void *)&err,
                    (void *)&limit_ns, (void *)&stall};
    return (int)cudaLaunchCooperativeKernel((const void *)k_potrf_tile, dim3(grid), dim3(POTRF_THREADS), args, PT_SMEM, s);
}

// log|A_i| = 2 sum log L_ii for every matrix of a batch (one CTA each, fixed order)
__global__ void __launch_bounds__(256) k_logdet_batched(const LEntry *__restrict__ e, int b, double *out) {
    __shared__ double red[256];
    const LEntry E = e[blockIdx.x];
    double s = 0.0;
    for (int64_t g = threadIdx.x; g < E.n; g += 256) {
        const int t = (int)(g / b), r = (int)(g % b);
        const double *D = E.W + ((int64_t)t * (t + 1) / 2 + t) * (int64_t)b * b;
        s += log(D[(int64_t)r * b + r]);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = 2.0 * red[0];
}

// identity padding of the last tile row of every ragged matrix (grid.z = matrix)
__global__ void k_fix_padding_batched(const LEntry *__restrict__ e, int b) {
    const LEntry E = e[blockIdx.z];
    const int j = blockIdx.y, i = E.nt - 1;
    if (j > i || E.n % b == 0) return;
    const int nv = (int)(E.n - (int64_t)i * b);
    double *T = E.W + ((int64_t)i * (i + 1) / 2 + j) * (int64_t)b * b;
    const int64_t bb = (int64_t)b * b;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < bb; x += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(x % b), c = (int)(x / b);
        if (j < i) {
            if (r >= nv) T[x] = 0.0;
        } else if (r >= nv || c >= nv) {
            T[x] = (r == c) ? 1.0 : 0.0;
        }
    }
}

void launch_logdet_batched(const LEntry *e, int count, int b, double *out, cudaStream_t s) {
    if (count > 0) k_logdet_batched<<<count, 256, 0, s>>>(e, b, out);
}
void launch_fix_padding_batched(const LEntry *e, int count, int ntmax, int b, cudaStream_t s) {
    if (count > 0) k_fix_padding_batched<<<dim3(16, ntmax, count), 256, 0, s>>>(e, b);
}


// ------------------------------------------------------------ grouped (batched) solves
__global__ void __launch_bounds__(256) k_fwd_diag_g(const SDiag *__restrict__ e, double *R, int b) {
    const SDiag E = e[blockIdx.y];
    fwd_diag_body(E.L, b, b, R + E.off + blockIdx.x * E.ldr);
}

template <int NQ>
__global__ void __launch_bounds__(256) k_fwd_update_g(const SUpd *__restrict__ u, double *R, int b, int nrhs) {
    const SUpd U = u[blockIdx.x];
    __shared__ double zs[128][16];
    __shared__ double red[64][17];
    const int tid = threadIdx.x, rr = tid & 63, part = tid >> 6;
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    for (int c0 = 0; c0 < b; c0 += 128) {
        const int nc = min(128, b - c0);          // a tile need not be a multiple of 128
        __syncthreads();
        for (int e = tid; e < 128 * nrhs; e += 256) {
            const int c = e % 128, q = e / 128;
            if (c < nc) zs[c][q] = R[U.src + q * U.ldr + c0 + c];
        }
        __syncthreads();
        for (int c = part; c < nc; c += 4) {
            const double l = U.L[(int64_t)(c0 + c) * b + U.r0 + rr];
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nrhs) acc[q] = fma(l, zs[c][q], acc[q]);
        }
    }
    part_reduce_sub(red, acc, nrhs, R + U.dst, U.ldr, 0);
}

__global__ void __launch_bounds__(256) k_bwd_diag_g(const SDiag *__restrict__ e, double *R, int b) {
    const SDiag E = e[blockIdx.y];
    bwd_diag_body(E.L, b, b, R + E.off + blockIdx.x * E.ldr);
}

template <int NQ>
__global__ void __launch_bounds__(256) k_bwd_update_g(const SUpd *__restrict__ u, double *R, int b, int nrhs) {
    const SUpd U = u[blockIdx.x];
    __shared__ double xs[64][16];
    __shared__ double S[64][65];
    const int tid = threadIdx.x, rr = tid & 63, part = tid >> 6;
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    for (int c0 = 0; c0 < b; c0 += 64) {
        __syncthreads();
        for (int idx = tid; idx < 4096; idx += 256) {
            const int c = idx & 63, r = idx >> 6;
            S[r][c] = U.L[(int64_t)(U.r0 + r) * b + c0 + c];
        }
        for (int e = tid; e < 64 * nrhs; e += 256) {
            const int c = e % 64, q = e / 64;
            xs[c][q] = R[U.src + q * U.ldr + c0 + c];
        }
        __syncthreads();
        for (int c = part; c < 64; c += 4) {
            const double l = S[rr][c];
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nrhs) acc[q] = fma(l, xs[c][q], acc[q]);
        }
    }
    part_reduce_sub(reinterpret_cast<double(*)[17]>(&S[0][0]), acc, nrhs, R + U.dst, U.ldr, 0);
}

// FP32 forms of the grouped substitution (the correction solves of a refined batched solve): the
// factor tiles are read in FP64 and rounded to FP32 on load, products and sums run on the FP32
// pipe (GB300 retires 64x more FP32 than FP64 operations per clock); the diagonal blocks keep
// FP64 arithmetic on the FP32 vectors.  Iterative refinement with FP64 residuals takes the
// result to FP64 accuracy: a correction needs only a few correct digits.
template <int NQ>
__device__ __forceinline__ void part_reduce_sub_f(float (*red)[17], const float (&acc)[NQ], int nrhs, float *R,
                                                  int64_t ldr) {
    const int tid = threadIdx.x, rr = tid & 63, part = tid >> 6;
    for (int p = 0; p < 4; ++p) {
        __syncthreads();
        if (part == p)
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nrhs) red[rr][q] = (p == 0) ? acc[q] : red[rr][q] + acc[q];
    }
    __syncthreads();
    for (int e = tid; e < 64 * nrhs; e += 256) {
        const int r = e % 64, q = e / 64;
        R[q * ldr + r] -= red[r][q];
    }
}
__global__ void __launch_bounds__(256) k_fwd_diag_gf(const SDiag *__restrict__ e, float *R, int b) {
    const SDiag E = e[blockIdx.y];
    fwd_diag_body(E.L, b, b, R + E.off + blockIdx.x * E.ldr);
}
__global__ void __launch_bounds__(256) k_bwd_diag_gf(const SDiag *__restrict__ e, float *R, int b) {
    const SDiag E = e[blockIdx.y];
    bwd_diag_body(E.L, b, b, R + E.off + blockIdx.x * E.ldr);
}
template <int NQ>
__global__ void __launch_bounds__(256) k_fwd_update_gf(const SUpd *__restrict__ u, float *R, int b, int nrhs) {
    const SUpd U = u[blockIdx.x];
    __shared__ float zs[128][17];
    __shared__ float red[64][17];
    const int tid = threadIdx.x, rr = tid & 63, part = tid >> 6;
    float acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.f;
    for (int c0 = 0; c0 < b; c0 += 128) {
        const int nc = min(128, b - c0);          // a tile need not be a multiple of 128
        __syncthreads();
        for (int e = tid; e < 128 * nrhs; e += 256) {
            const int c = e % 128, q = e / 128;
            if (c < nc) zs[c][q] = R[U.src + q * U.ldr + c0 + c];
        }
        __syncthreads();
        for (int c = part; c < nc; c += 4) {
            const float l = (float)U.L[(int64_t)(c0 + c) * b + U.r0 + rr];
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nrhs) acc[q] = fmaf(l, zs[c][q], acc[q]);
        }
    }
    part_reduce_sub_f(red, acc, nrhs, R + U.dst, U.ldr);
}
template <int NQ>
__global__ void __launch_bounds__(256) k_bwd_update_gf(const SUpd *__restrict__ u, float *R, int b, int nrhs) {
    const SUpd U = u[blockIdx.x];
    __shared__ float xs[64][17];
    __shared__ float S[64][65];
    __shared__ float red[64][17];
    const int tid = threadIdx.x, rr = tid & 63, part = tid >> 6;
    float acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.f;
    for (int c0 = 0; c0 < b; c0 += 64) {
        __syncthreads();
        for (int idx = tid; idx < 4096; idx += 256) {
            const int c = idx & 63, r = idx >> 6;
            S[r][c] = (float)U.L[(int64_t)(U.r0 + r) * b + c0 + c];
        }
        for (int e = tid; e < 64 * nrhs; e += 256) {
            const int c = e % 64, q = e / 64;
            xs[c][q] = R[U.src + q * U.ldr + c0 + c];
        }
        __syncthreads();
        for (int c = part; c < 64; c += 4) {
            const float l = S[rr][c];
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nrhs) acc[q] = fmaf(l, xs[c][q], acc[q]);
        }
    }
    part_reduce_sub_f(red, acc, nrhs, R + U.dst, U.ldr);
}
__global__ void k_to_f32(const double *__restrict__ x, float *__restrict__ y, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = (float)x[i];
}
__global__ void k_add_f32(double *__restrict__ x, const float *__restrict__ d, int64_t n, int assign) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x[i] = assign ? (double)d[i] : x[i] + (double)d[i];
}

template <int NQ>
__global__ void __launch_bounds__(256)
k_symv_g(const SRes *__restrict__ rs, int b, const double *X, const double *B, double *R, int nrhs, int absmode) {
    const SRes Q = rs[blockIdx.x];
    __shared__ double xs[64][16];
    __shared__ double S[64][65];
    const int i = Q.i, r0 = Q.r0;
    const int tid = threadIdx.x, rr = tid & 63, part = tid >> 6;
    const int64_t bb = (int64_t)b * b;
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    for (int j = 0; j < Q.nt; ++j) {
        const bool lower = j <= i;
        const double *T = lower ? Q.A + ((int64_t)i * (i + 1) / 2 + j) * bb : Q.A + ((int64_t)j * (j + 1) / 2 + i) * bb;
        for (int c0 = 0; c0 < b; c0 += 64) {
            __syncthreads();
            for (int idx = tid; idx < 4096; idx += 256) {
                const int lo = idx & 63, hi = idx >> 6;
                double v;
                int64_t gr, gc;
                if (lower) {
                    v = T[(int64_t)(c0 + hi) * b + r0 + lo];
                    gr = (int64_t)i * b + r0 + lo; gc = (int64_t)j * b + c0 + hi;
                    if (gr >= Q.n || gc >= Q.n) v = 0.0;
                    S[lo][hi] = absmode ? fabs(v) : v;
                } else {
                    v = T[(int64_t)(r0 + hi) * b + c0 + lo];
                    gr = (int64_t)i * b + r0 + hi; gc = (int64_t)j * b + c0 + lo;
                    if (gr >= Q.n || gc >= Q.n) v = 0.0;
                    S[hi][lo] = absmode ? fabs(v) : v;
                }
            }
            for (int e = tid; e < 64 * nrhs; e += 256) {
                const int c = e % 64, q = e / 64;
                const int64_t g = (int64_t)j * b + c0 + c;
                xs[c][q] = (g < Q.n) ? (X ? X[Q.xo + q * Q.ldr + g] : 1.0) : 0.0;
            }
            __syncthreads();
            for (int c = part; c < 64; c += 4) {
                const double l = S[rr][c];
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (q < nrhs) acc[q] = fma(l, xs[c][q], acc[q]);
            }
        }
    }
    double(*red)[17] = reinterpret_cast<double(*)[17]>(&S[0][0]);
    for (int p = 0; p < 4; ++p) {
        __syncthreads();
        if (part == p)
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (q < nrhs) red[rr][q] = (p == 0) ? acc[q] : red[rr][q] + acc[q];
    }
    __syncthreads();
    for (int e = tid; e < 64 * nrhs; e += 256) {
        const int r = e % 64, q = e / 64;
        const int64_t g = (int64_t)i * b + r0 + r;
        double out = 0.0;
        if (g < Q.n) out = absmode ? red[r][q] : B[Q.bo + q * Q.ldr + g] - red[r][q];
        R[Q.ro + q * Q.ldr + g] = out;
    }
}

__global__ void k_colmax_g(const SMax *__restrict__ m, const double *V, int nrhs, double *out) {
    const SMax M = m[blockIdx.y];
    for (int c = 0; c < nrhs; ++c) {
        double mx = 0.0;
        for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < M.n; r += (int64_t)gridDim.x * blockDim.x)
            mx = fmax(mx, fabs(V[M.off + c * M.ldr + r]));
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0)
            atomicMax(reinterpret_cast<unsigned long long *>(out + M.out + c), (unsigned long long)__double_as_longlong(mx));
    }
}

__global__ void k_axpy_flat(double *X, const double *D, int64_t count) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        X[e] += D[e];
}

// one CTA per matrix: out[M.out] = u . v over its n entries (fixed order)
__global__ void __launch_bounds__(256) k_dots_g(const SMax *__restrict__ m, const double *u, const double *v, double *out) {
    const SMax M = m[blockIdx.x];
    __shared__ double red[256];
    double s = 0.0;
    for (int64_t r = threadIdx.x; r < M.n; r += 256) s = fma(u[M.off + r], v[M.off + r], s);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[M.out] = red[0];
}

void launch_fwd_diag_g(const SDiag *e, int ne, double *R, int b, int nrhs, cudaStream_t s) {
    if (ne > 0) k_fwd_diag_g<<<dim3(nrhs, ne), 256, 0, s>>>(e, R, b);
}
void launch_fwd_update_g(const SUpd *u, int nu, double *R, int b, int nrhs, cudaStream_t s) {
    if (nu > 0) NQ_DISPATCH(nrhs, k_fwd_update_g, nu, 256, 0, s, u, R, b, nrhs);
}
void launch_bwd_diag_g(const SDiag *e, int ne, double *R, int b, int nrhs, cudaStream_t s) {
    if (ne > 0) k_bwd_diag_g<<<dim3(nrhs, ne), 256, 0, s>>>(e, R, b);
}
void launch_bwd_update_g(const SUpd *u, int nu, double *R, int b, int nrhs, cudaStream_t s) {
    if (nu > 0) NQ_DISPATCH(nrhs, k_bwd_update_g, nu, 256, 0, s, u, R, b, nrhs);
}
void launch_fwd_diag_gf(const SDiag *e, int ne, float *R, int b, int nrhs, cudaStream_t s) {
    if (ne > 0) k_fwd_diag_gf<<<dim3(nrhs, ne), 256, 0, s>>>(e, R, b);
}
void launch_fwd_update_gf(const SUpd *u, int nu, float *R, int b, int nrhs, cudaStream_t s) {
    if (nu > 0) NQ_DISPATCH(nrhs, k_fwd_update_gf, nu, 256, 0, s, u, R, b, nrhs);
}
void launch_bwd_diag_gf(const SDiag *e, int ne, float *R, int b, int nrhs, cudaStream_t s) {
    if (ne > 0) k_bwd_diag_gf<<<dim3(nrhs, ne), 256, 0, s>>>(e, R, b);
}
void launch_bwd_update_gf(const SUpd *u, int nu, float *R, int b, int nrhs, cudaStream_t s) {
    if (nu > 0) NQ_DISPATCH(nrhs, k_bwd_update_gf, nu, 256, 0, s, u, R, b, nrhs);
}
void launch_to_f32(const double *x, float *y, int64_t n, cudaStream_t s) {
    if (n > 0) k_to_f32<<<608, 256, 0, s>>>(x, y, n);
}
void launch_add_f32(double *x, const float *d, int64_t n, int assign, cudaStream_t s) {
    if (n > 0) k_add_f32<<<608, 256, 0, s>>>(x, d, n, assign);
}
void launch_symv_g(const SRes *r, int nr, int b, const double *X, const double *B, double *R, int nrhs, int absmode,
                   cudaStream_t s) {
    if (nr > 0) NQ_DISPATCH(nrhs, k_symv_g, nr, 256, 0, s, r, b, X, B, R, nrhs, absmode);
}
void launch_colmax_g(const SMax *m, int nm, const double *V, int nrhs, double *out, cudaStream_t s) {
    if (nm > 0) k_colmax_g<<<dim3(8, nm), 256, 0, s>>>(m, V, nrhs, out);
}
void launch_axpy_flat(double *X, const double *D, int64_t count, cudaStream_t s) {
    k_axpy_flat<<<1024, 256, 0, s>>>(X, D, count);
}
void launch_dots_g(const SMax *m, int nm, const double *u, const double *v, double *out, cudaStream_t s) {
    if (nm > 0) k_dots_g<<<nm, 256, 0, s>>>(m, u, v, out);
}

// ---------------------------------------------------------------------------- launchers

void launch_dgemm_update(const DJob *jobs, const DItem *items, int nitems, int ld, double *partials,
                         const int *status, cudaStream_t s) {
    if (nitems > 0) k_dgemm_update<<<nitems, 256, 0, s>>>(jobs, items, ld, partials, status);
}
void launch_dgemm_reduce(const DRed *reds, int nreds, int ld, const double *partials, const int *status,
                         cudaStream_t s) {
    if (nreds > 0) k_dgemm_reduce<<<nreds, 256, 0, s>>>(reds, ld, partials, status);
}
void launch_potrf_block(double *D, int ld, int col0, int *status, cudaStream_t s) {
    k_potrf_block<<<1, POTRF_THREADS, 0, s>>>(D, ld, col0, status);
}
void launch_trsm_rows(double *P, const double *L, int ld, int rows, const int *status, cudaStream_t s) {
    if (rows > 0) k_trsm_rows<<<rows / PANEL_ROWS, 256, 0, s>>>(P, L, ld, status);
}
void launch_trsm_strips(const TStrip *strips, int nstrips, int rows, int ld, int b, const int *status, cudaStream_t s) {
    if (nstrips <= 0) return;
    if (rows == SMALL_STRIP) {
        k_trsm_strips16<<<nstrips, 256, 0, s>>>(strips, ld, b, status);
        return;
    }
    const size_t smem = (32 * 64 + 2 * 64 * 65 + 64) * sizeof(double);
    static std::atomic<unsigned long long> attr{0};
    if (attrs_pending(attr)) {
        cudaFuncSetAttribute(k_trsm_strips, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        mark_attrs_set(attr);
    }
    k_trsm_strips<<<nstrips, 256, smem, s>>>(strips, ld, b, status);
}
void launch_logdet(const double *W, int nt, int b, int64_t n, double *out, cudaStream_t s) {
    (void)nt;
    k_logdet<<<1, 1024, 0, s>>>(W, b, n, out);
}
void launch_fix_padding(double *W, int nt, int b, int64_t n, cudaStream_t s) {
    if (n % b == 0) return;
    k_fix_padding<<<dim3(64, nt), 256, 0, s>>>(W, nt, b, n);
}
void launch_zero_upper_diag(double *W, int nt, int b, int64_t n, cudaStream_t s) {
    k_zero_upper_diag<<<dim3(64, (n % b) ? 2 * nt - 1 : nt), 256, 0, s>>>(W, nt, b, n);
}
void launch_symv_resid(const double *A, int nt, int b, int64_t n, const double *X, int64_t ldx,
                       const double *B, int64_t ldb, double *R, int64_t ldr, int nrhs, int absmode,
                       cudaStream_t s) {
    const auto al16 = [](const void *p) { return ((uintptr_t)p & 15) == 0; };
    if (nrhs == 1 && al16(A) && al16(X) && b % 64 == 0) {      // 16-byte loads of A and x
        if (absmode)
            k_symv1<true><<<nt * (b / 64), 256, 0, s>>>(A, nt, b, n, X, nullptr, R);
        else
            k_symv1<false><<<nt * (b / 64), 256, 0, s>>>(A, nt, b, n, X, B, R);
        return;
    }
    // groups of eight columns; a rest of one to four has a kernel of its own width
    const int rest = nrhs % 8 <= 4 ? nrhs % 8 : 0, main = nrhs - rest, rows = nt * (b / 64);
    if (main)
        k_symv_resid<8><<<rows * ((main + 7) / 8), 256, 0, s>>>(A, nt, b, n, X, ldx, B, ldb, R, ldr, main, absmode);
    if (!rest) return;
    X += main * ldx;
    B += main * ldb;
    R += main * ldr;
    if (main && rest == 1) launch_symv_resid(A, nt, b, n, X, ldx, B, ldb, R, ldr, 1, absmode, s);
    else if (rest == 1) k_symv_resid<1><<<rows, 256, 0, s>>>(A, nt, b, n, X, ldx, B, ldb, R, ldr, 1, absmode);
    else k_symv_resid<4><<<rows, 256, 0, s>>>(A, nt, b, n, X, ldx, B, ldb, R, ldr, rest, absmode);
}
void launch_colmax_abs(const double *V, int64_t ld, int64_t n, int ncols, double *out, cudaStream_t s) {
    k_colmax_abs<<<dim3(64, ncols), 256, 0, s>>>(V, ld, n, out);
}
void launch_axpy_cols(double *X, int64_t ldx, const double *D, int64_t ldd, int64_t n, int ncols, cudaStream_t s) {
    k_axpy_cols<<<dim3(64, ncols), 256, 0, s>>>(X, ldx, D, ldd, n);
}
__global__ void __launch_bounds__(1024) k_dot(const double *u, const double *v, int64_t n, double *out) {
    __shared__ double red[1024];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += 1024) s = fma(u[i], v[i], s);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 512; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

void launch_dot(const double *u, const double *v, int64_t n, double *out, cudaStream_t s) {
    k_dot<<<1, 1024, 0, s>>>(u, v, n, out);
}

void launch_dot_self(const double *v, int64_t n, double *out, cudaStream_t s) {
    k_dot_self<<<1, 1024, 0, s>>>(v, n, out);
}

// ------------------------------------------------------------- tile-pointer variants
// Used by the out-of-core executor, whose tiles live in cache slots at arbitrary
// addresses: the job comes by value and the grid is the 64 x 64 block grid.
__global__ void __launch_bounds__(256, 2) k_dgemm_tile(const DJob job, int ld) {
    const int bi = blockIdx.x, bj = blockIdx.y;
    if (job.lower && bi < bj) return;
    __shared__ double Xs[16][64], Ys[16][64];
    double acc[4][4] = {};
    dgemm_block(acc, job.X + bi * 64, job.Y + bj * 64, ld, 0, job.K, Xs, Ys);
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    double *C = job.C + (int64_t)bj * 64 * ld + bi * 64;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) C[(int64_t)(ty + 16 * j) * ld + tx + 16 * i] -= acc[i][j];
}

// TRSM of up to TG_MAX tiles at C[0..] with the same L_kk at L (one CTA per 64-row strip;
// grid b/64 x tiles).
struct TGroup {
    double *C[TG_MAX];
};
__global__ void __launch_bounds__(256, 2)
k_trsm_tile(const __grid_constant__ TGroup g, const double *L, int ld, int b, const int *status) {
    if (failed(status)) return;
    double *C = g.C[blockIdx.y];
    extern __shared__ double smem[];
    double(*Xs)[64] = reinterpret_cast<double(*)[64]>(smem);
    double(*Ys)[64] = reinterpret_cast<double(*)[64]>(smem + 16 * 64);
    double(*Ls)[65] = reinterpret_cast<double(*)[65]>(smem + 32 * 64);
    double(*Ss)[65] = reinterpret_cast<double(*)[65]>(smem + 32 * 64 + 64 * 65);
    double *rinv = smem + 32 * 64 + 2 * 64 * 65;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double *X = C + blockIdx.x * 64;
    for (int jb = 0; jb < b / 64; ++jb) {
        double acc[4][4] = {};
        dgemm_block(acc, X, L + jb * 64, ld, 0, jb * 64, Xs, Ys);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                Ss[tx + 16 * i][ty + 16 * j] = X[(int64_t)(jb * 64 + ty + 16 * j) * ld + tx + 16 * i] - acc[i][j];
        for (int idx = tid; idx < 4096; idx += 256) {
            const int r = idx & 63, c = idx >> 6;
            Ls[r][c] = (r >= c) ? L[(int64_t)(jb * 64 + c) * ld + jb * 64 + r] : 0.0;
        }
        __syncthreads();
        if (tid < 64) rinv[tid] = 1.0 / Ls[tid][tid];
        __syncthreads();
        strip_solve<64>(Ss, Ls, rinv);
        for (int idx = tid; idx < 4096; idx += 256) {
            const int r = idx & 63, c = idx >> 6;
            X[(int64_t)(jb * 64 + c) * ld + r] = Ss[r][c];
        }
        __syncthreads();
    }
}

// Mixed maps: Y = L^{-1} for a lower-triangular b x b tile L (column-major, ld = b), by forward
// substitution L y_c = e_c column by column, two columns a CTA (column c costs (b - c)^2 / 2
// multiply-adds, the longest come first).  For each 64-row block from the columns' own on, the product
// with the solved rows, kept in shared memory, is followed by the block's triangle: a warp per
// column, y_j and with it the next row by shuffle, the division in integer arithmetic (the same
// rounding, fixed_exp.h).
// In core only, and for bits rather than accuracy: the products with Y of a mixed factorization keep 10, 6
// or 4 of its digit planes, so what they cut off, and with it the last bit of a stored FP32, FP16 or FP8
// value here and there, follows the inverse's own rounding, and this substitution, every element's
// multiply-adds in ascending order, keeps the factors of a map as they have been.  The doubling of
// k_bgemm.cu, several times as fast, serves all-FP64 maps and every map out of core, where the planes are
// base 256 and the factor is another one within the accuracy level anyway.  Its inverse is no less exact (a
// CPU model on Matern tiles of 256 and 512, condition of L_kk 15 to 7e6: the largest entry of Y L - I is 0.09
// to 0.7 of this one's, that of L Y - I 0.6 to 30 times it, both far below the planes' 2^-41), and the mixed
// factors out of core are 0.82 to 0.999 times as far from 64 bits as with this one and base 16.
// What bounds it: the FP64 pipe (b^3 / 6 multiply-adds, 2.7 ms for a tile of 2048).  So L's blocks
// arrive one ahead of their use, and the SM's other CTAs run while one is on its chain.  A tile of
// 2048: 4.24 ms with four columns and 256 threads, barriers in the triangle and L read where it is
// used, 3.23 ms here.
constexpr int TRINV_COLS = 2, TRINV_THREADS = 128;
struct TrinvDiv {
    unsigned long long m, v;
    int e, ok;
};
static size_t trinv_smem(int b) {
    return (2 * 4096 + (size_t)b * TRINV_COLS + 64 * TRINV_COLS) * sizeof(double) + 64 * sizeof(TrinvDiv);
}
// RN(z / l), l the divisor D was made from
__device__ __forceinline__ double trinv_div(double z, double l, const TrinvDiv &D) {
    const unsigned long long w = (unsigned long long)__double_as_longlong(z);
    const int e = (int)(w >> 52) & 2047;
    if (w == 0 && D.ok) return z;
    if (!D.ok || e <= 400 || e >= 1646) return z / l;      // quotients stay normal in between
    fx::Num h;
    h.m = (w & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    h.e = e - 1075;
    fx::Divisor a;
    a.m = D.m;
    a.v = D.v;
    a.e = D.e;
    return __longlong_as_double(__double_as_longlong(fx::value(fx::div_rn(h, a))) | (long long)(w & (1ull << 63)));
}
// block (ib, jb) of L into S[column][row]
__device__ __forceinline__ void trinv_load(double *S, const double *__restrict__ L, int b, int ib, int jb) {
#pragma unroll 8
    for (int i = threadIdx.x; i < 4096; i += TRINV_THREADS)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(S + i)),
                     "l"(L + (int64_t)(jb * 64 + (i >> 6)) * b + ib * 64 + (i & 63))
                     : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}
// several tiles at once (grid.y = entry): the diagonal tiles of a batch's column
__global__ void __launch_bounds__(TRINV_THREADS) k_trinv_batched(const TEntry *__restrict__ e, int b) {
    extern __shared__ double tsm[];
    double *S = tsm;                                          // two 64 x 64 blocks of L
    double *Ys = tsm + 2 * 4096;                              // the solved rows, column by column
    double *Acc = Ys + (size_t)b * TRINV_COLS;                // one block's rows
    TrinvDiv *Dv = reinterpret_cast<TrinvDiv *>(Acc + 64 * TRINV_COLS);
    const double *__restrict__ L = e[blockIdx.y].L;
    const int tid = threadIdx.x, r = tid & 63, cg = tid >> 6, warp = tid >> 5, lane = tid & 31;
    const int c = blockIdx.x * TRINV_COLS + cg, ib0 = (int)blockIdx.x * TRINV_COLS / 64;
    double *Y = e[blockIdx.y].Y + (int64_t)c * b, *Yc = Ys + (size_t)cg * b;
    for (int i = r; i < ib0 * 64; i += 64) Y[i] = 0.0;
    trinv_load(S, L, b, ib0, ib0);
    int cur = 0;
    for (int ib = ib0; ib < b / 64; ++ib) {
        double a = (ib * 64 + r == c) ? 1.0 : 0.0;
        for (int jb = ib0; jb <= ib; ++jb, cur ^= 1) {
            const int ni = jb < ib ? ib : ib + 1, nj = jb < ib ? jb + 1 : ib0;
            // the other buffer's readers passed the barrier that ended their step
            if (ni < b / 64) {
                trinv_load(S + (cur ^ 1) * 4096, L, b, ni, nj);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            const double *B = S + cur * 4096;
            if (jb < ib) {
#pragma unroll 16
                for (int l = 0; l < 64; ++l) a = fma(-B[l * 64 + r], Yc[jb * 64 + l], a);
            } else {
                Acc[cg * 64 + r] = a;
                if (cg == 0) {
                    const double d = B[r * 65];
                    const int x = (int)((unsigned long long)__double_as_longlong(d) >> 52);     // sign included
                    TrinvDiv D;
                    D.ok = x > 400 && x < 1646;
                    const fx::Divisor q = fx::make_divisor(D.ok ? d : 1.0);
                    D.m = q.m;
                    D.v = q.v;
                    D.e = q.e;
                    Dv[r] = D;
                }
                __syncthreads();
                if (warp < TRINV_COLS) {
                    double z0 = Acc[warp * 64 + lane], z1 = Acc[warp * 64 + lane + 32];
                    for (int j = 0; j < 32; ++j) {
                        const double y = trinv_div(__shfl_sync(0xffffffffu, z0, j), B[j * 65], Dv[j]);
                        if (lane == j) z0 = y;
                        if (lane > j) z0 = fma(-B[j * 64 + lane], y, z0);
                        z1 = fma(-B[j * 64 + lane + 32], y, z1);
                    }
                    for (int j = 32; j < 64; ++j) {
                        const double y = trinv_div(__shfl_sync(0xffffffffu, z1, j - 32), B[j * 65], Dv[j]);
                        if (lane == j - 32) z1 = y;
                        if (lane > j - 32) z1 = fma(-B[j * 64 + lane + 32], y, z1);
                    }
                    double *out = Ys + (size_t)warp * b + ib * 64;
                    out[lane] = z0;
                    out[lane + 32] = z1;
                }
                __syncthreads();
                Y[ib * 64 + r] = Yc[ib * 64 + r];
            }
            __syncthreads();
        }
    }
}

// sum of log of the nv leading diagonal entries of one tile, fixed order, into *out
__global__ void __launch_bounds__(256) k_logdiag_tile(const double *D, int b, int nv, double *out) {
    __shared__ double red[256];
    double s = 0.0;
    for (int r = threadIdx.x; r < nv; r += 256) s += log(D[(int64_t)r * b + r]);
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0];
}

// padding of one tile of the last tile row: rows >= nv zero (off-diagonal), identity
// outside the nv x nv block (diagonal)
__global__ void k_fix_padding_tile(double *T, int b, int nv, int diag) {
    const int64_t bb = (int64_t)b * b;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < bb; e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e % b), c = (int)(e / b);
        if (!diag) {
            if (r >= nv) T[e] = 0.0;
        } else if (r >= nv || c >= nv) {
            T[e] = (r == c) ? 1.0 : 0.0;
        }
    }
}

// r_i -= L_ij z_j for one tile L_ij (ptr).  What bounds these two: reading the tile, if enough CTAs
// share it.  16 rows a CTA (a column's 128 bytes at a time), 16 threads a row, each with its next
// eight elements in flight while z is staged; backwards a warp per row of L^T.  A tile
// of 1024, one column: forward 39 us with 64 rows a CTA, 12.5 us here; backward 62 us with 64 rows
// staged in shared memory.
constexpr int TU_ROWS = 16, TU_COLS = 128;
template <int NQ>
__global__ void __launch_bounds__(256)
k_fwd_update_tile(const double *L, int b, int i, int j, double *R, int64_t ldr, int nrhs) {
    __shared__ double buf[16 * NQ * (TU_ROWS + 1)];
    double(*zs)[NQ] = reinterpret_cast<double(*)[NQ]>(buf);                                    // TU_COLS rows of z, then
    double(*red)[NQ][TU_ROWS + 1] = reinterpret_cast<double(*)[NQ][TU_ROWS + 1]>(buf);         // the 16 parts' sums
    static_assert(TU_COLS <= 16 * (TU_ROWS + 1), "z fits their place");
    const int r0 = blockIdx.x * TU_ROWS;
    const int tid = threadIdx.x, rr = tid & 15, part = tid >> 4;
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
    for (int c0 = 0; c0 < b; c0 += TU_COLS) {
        const int nc = min(TU_COLS, b - c0);
        double l[TU_COLS / 16];
#pragma unroll
        for (int u = 0; u < TU_COLS / 16; ++u)
            l[u] = part + 16 * u < nc ? L[(int64_t)(c0 + part + 16 * u) * b + r0 + rr] : 0.0;
        __syncthreads();
        for (int e = tid; e < TU_COLS * NQ; e += 256) {
            const int c = e % TU_COLS, q = e / TU_COLS;
            zs[c][q] = c < nc && q < nrhs ? R[q * ldr + (int64_t)j * b + c0 + c] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < TU_COLS / 16; ++u)
#pragma unroll
            for (int q = 0; q < NQ; ++q) acc[q] = fma(l[u], zs[part + 16 * u][q], acc[q]);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NQ; ++q) red[part][q][rr] = acc[q];
    __syncthreads();
    for (int e = tid; e < TU_ROWS * nrhs; e += 256) {
        const int r = e % TU_ROWS, q = e / TU_ROWS;
        double sum = 0.0;
#pragma unroll
        for (int p = 0; p < 16; ++p) sum += red[p][q][r];
        R[q * ldr + (int64_t)i * b + r0 + r] -= sum;
    }
}

// z_i -= L_ji^T x_j for one tile L_ji (ptr)
template <int NQ>
__global__ void __launch_bounds__(256)
k_bwd_update_tile(const double *L, int b, int i, int j, double *R, int64_t ldr, int nrhs) {
    const int lane = threadIdx.x & 31, r = blockIdx.x * 8 + (threadIdx.x >> 5);
    const double *l = L + (int64_t)r * b, *x = R + (int64_t)j * b;
    double acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = 0.0;
#pragma unroll 8
    for (int c = lane; c < b; c += 32) {
        const double v = l[c];
#pragma unroll
        for (int q = 0; q < NQ; ++q)
            if (q < nrhs) acc[q] = fma(v, __ldcg(x + q * ldr + c), acc[q]);
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
        if (lane == 0 && q < nrhs) R[q * ldr + (int64_t)i * b + r] -= acc[q];
    }
}

void launch_dgemm_tile(const DJob &job, int ld, cudaStream_t s) {
    k_dgemm_tile<<<dim3(job.M / 64, job.N / 64), 256, 0, s>>>(job, ld);
}
static size_t trsm_tile_smem() {
    const size_t smem = (32 * 64 + 2 * 64 * 65 + 64) * sizeof(double);
    static std::atomic<unsigned long long> attr{0};
    if (attrs_pending(attr)) {
        cudaFuncSetAttribute(k_trsm_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        mark_attrs_set(attr);
    }
    return smem;
}
void launch_trsm_tile(double *C, const double *L, int ld, int b, const int *status, cudaStream_t s) {
    launch_trsm_group(&C, 1, L, ld, b, status, s);
}
void launch_trsm_group(double *const *C, int ntiles, const double *L, int ld, int b, const int *status,
                       cudaStream_t s) {
    if (ntiles <= 0) return;
    const size_t smem = trsm_tile_smem();
    TGroup g{};
    for (int t = 0; t < ntiles; ++t) g.C[t] = C[t];
    k_trsm_tile<<<dim3(b / 64, ntiles), 256, smem, s>>>(g, L, ld, b, status);
}
void launch_trinv_columns(const TEntry *e, int n, int b, cudaStream_t s) {
    if (n <= 0) return;
    static std::atomic<unsigned long long> attr{0};
    if (attrs_pending(attr)) {     // sized for the largest tile it serves (b <= 2048)
        cudaFuncSetAttribute(k_trinv_batched, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)trinv_smem(2048));
        mark_attrs_set(attr);
    }
    k_trinv_batched<<<dim3(b / TRINV_COLS, n), TRINV_THREADS, trinv_smem(b), s>>>(e, b);
}
void launch_logdiag_tile(const double *D, int b, int nv, double *out, cudaStream_t s) {
    k_logdiag_tile<<<1, 256, 0, s>>>(D, b, nv, out);
}
void launch_fix_padding_tile(double *T, int b, int nv, int diag, cudaStream_t s) {
    k_fix_padding_tile<<<64, 256, 0, s>>>(T, b, nv, diag);
}
void launch_fwd_update_tile(const double *L, int b, int i, int j, double *R, int64_t ldr, int nrhs, cudaStream_t s) {
    NQ_DISPATCH(nrhs, k_fwd_update_tile, b / TU_ROWS, 256, 0, s, L, b, i, j, R, ldr, nrhs);
}
void launch_bwd_update_tile(const double *L, int b, int i, int j, double *R, int64_t ldr, int nrhs, cudaStream_t s) {
    NQ_DISPATCH(nrhs, k_bwd_update_tile, b / 8, 256, 0, s, L, b, i, j, R, ldr, nrhs);
}

}  // namespace tc
