// Input preparation on the device: the Matern covariance of Eq. 2 (Section III-D) written
// straight into the lower tile layout, and the per-tile sums of squares behind the
// precision criterion of Section IV-C: integer work bounds the first, the FP64 pipe and HBM the
// second (at the kernels below).
#include "tc_internal.h"

#include <algorithm>
#include <cooperative_groups.h>

#define FIXED_FN __host__ __device__ __forceinline__
#include "fixed_exp.h"

#ifndef MATERN_FN
#define MATERN_FN __host__ __device__
#endif

namespace tc {

// ---------------------------------------------------------------- K_nu for any nu > 0
// Eq. 2 for a smoothness that is not a half integer needs the modified Bessel function of the
// second kind.  With nu = mu + m, |mu| <= 1/2, K_mu and K_{mu+1} come from
//   x <= 2: Temme's power series (N. M. Temme, J. Comput. Phys. 19 (1975) 324-337);
//   x >  2: Temme's normalising sum  sum_k C_k U_k = (2x)^-(mu+1/2)  over the confluent
//           functions U_k = U(mu+1/2+k, 2mu+1, 2x), whose ratios are the minimal solution of
//           their three-term recurrence, taken by Miller's backward recurrence (Gautschi,
//           SIAM Rev. 9 (1967) 24-82);
// and K_{mu+j+1} = K_{mu+j-1} + 2(mu+j)/x K_{mu+j} (stable upwards) reaches nu.

// g1 = (1/Gamma(1-mu) - 1/Gamma(1+mu)) / (2mu) and g2 = (1/Gamma(1-mu) + 1/Gamma(1+mu)) / 2
// for |mu| <= 1/2, from the odd and even parts of the Taylor series of 1/Gamma(1+z) at 0
// (Abramowitz & Stegun 6.1.34 lists it as the series of 1/Gamma(z), shifted by one power).
// Twenty-two terms leave a tail below 1e-18 at |z| = 1/2, and mu -> 0 needs no limit.
MATERN_FN inline void temme_gammas(double mu, double &g1, double &g2) {
    const double m2 = mu * mu;
    g1 = -(5.7721566490153286e-1 + m2 * (-4.2002635034095236e-2 + m2 * (-4.2197734555544337e-2 +
           m2 * (7.2189432466630995e-3 + m2 * (-2.1524167411495097e-4 + m2 * (-2.0134854780788239e-5 +
           m2 * (1.1330272319816959e-6 + m2 * (6.1160951044814158e-9 + m2 * (-1.1812745704870201e-9 +
           m2 * (7.7822634399050713e-12 + m2 * 5.1003702874544760e-13))))))))));
    g2 = 1.0 + m2 * (-6.5587807152025388e-1 + m2 * (1.6653861138229149e-1 + m2 * (-9.6219715278769736e-3 +
         m2 * (-1.1651675918590651e-3 + m2 * (1.2805028238811619e-4 + m2 * (-1.2504934821426707e-6 +
         m2 * (-2.0563384169776071e-7 + m2 * (5.0020076444692229e-9 + m2 * (1.0434267116911005e-10 +
         m2 * -3.6968056186422057e-12)))))))));
}

// Per-call constants of the Matern correlation for smoothness nu: m = floor(nu + 1/2),
// mu = nu - m, Temme's g1, g2 and pre = 2^(1-nu) / Gamma(nu), with
// Gamma(nu) = Gamma(1+mu) (mu+1) ... (mu+m-1), or Gamma(1+mu)/mu when m = 0; and what the two
// evaluations below would otherwise divide by for every element (an FP64 division is 7 FP64
// operations): made once, on the host.
struct MaternNu {
    static constexpr int KS = 24, KR = 82;      // terms of the series, of the normalising sum
    double nu, mu, g1, g2, pre;
    double fac, ip, iq;                         // mu pi / sin(mu pi), Gamma(1+mu) / 2, Gamma(1-mu) / 2
    double r2[KS], rm[KS], rp[KS], rf[KS];      // 1/(k^2 - mu^2), prod 1/(j - mu), prod 1/(j + mu), 1/k!
    double a[KR], c[KR];                        // a_k = (k+1/2)^2 - mu^2, C_k = C_{k-1} a_{k-1} / k
    int m;
};

MATERN_FN inline MaternNu matern_nu(double nu) {
    MaternNu c;
    c.nu = nu;
    c.m = (int)floor(nu + 0.5);
    c.mu = nu - c.m;
    temme_gammas(c.mu, c.g1, c.g2);
    c.ip = 0.5 / (c.g2 - c.mu * c.g1);          // 1/Gamma(1+mu) = g2 - mu g1
    c.iq = 0.5 / (c.g2 + c.mu * c.g1);          // 1/Gamma(1-mu) = g2 + mu g1
    double gam = 2.0 * c.ip;
    if (c.m == 0) gam /= c.mu;
    for (int j = 1; j < c.m; ++j) gam *= c.mu + j;
    c.pre = exp2(1.0 - nu) / gam;
    c.fac = (c.mu == 0.0) ? 1.0 : (3.141592653589793 * c.mu) / sin(3.141592653589793 * c.mu);
    const double m2 = c.mu * c.mu;
    c.r2[0] = 0.0;
    c.rm[0] = c.rp[0] = c.rf[0] = 1.0;
    for (int k = 1; k < MaternNu::KS; ++k) {
        c.r2[k] = 1.0 / ((double)k * k - m2);
        c.rm[k] = c.rm[k - 1] / (k - c.mu);
        c.rp[k] = c.rp[k - 1] / (k + c.mu);
        c.rf[k] = c.rf[k - 1] / k;
    }
    c.c[0] = 1.0;
    for (int k = 0; k < MaternNu::KR; ++k) {
        c.a[k] = (k + 0.5) * (k + 0.5) - m2;
        if (k > 0) c.c[k] = c.c[k - 1] * (c.a[k - 1] / k);
    }
    return c;
}

// sinh(s) / s from e = exp(s) and 1/e, the Taylor series where the difference would cancel
MATERN_FN inline double sinh_ratio(double s, double e, double ei) {
    if (fabs(s) > 0.5) return 0.5 * (e - ei) / s;
    const double t = s * s;
    return 1.0 + t * (1.0 / 6.0) * (1.0 + t * (1.0 / 20.0) * (1.0 + t * (1.0 / 42.0) * (1.0 + t * (1.0 / 72.0) *
               (1.0 + t * (1.0 / 110.0) * (1.0 + t * (1.0 / 156.0) * (1.0 + t * (1.0 / 210.0)))))));
}

// K_mu(x), K_{mu+1}(x) for |mu| <= 1/2, 0 < x <= 2.  With c_k = (x^2/4)^k / k!:
//   K_mu = sum c_k f_k,  K_{mu+1} = (2/x) sum c_k (p_k - k f_k),
//   f_k = (k f_{k-1} + p_{k-1} + q_{k-1}) / (k^2 - mu^2),  p_k = p_{k-1}/(k-mu),  q_k = q_{k-1}/(k+mu),
//   p_0 = (x/2)^-mu Gamma(1+mu) / 2,  q_0 = (x/2)^mu Gamma(1-mu) / 2,
//   f_0 = (mu pi / sin(mu pi)) (cosh(s) g1 + sinh(s)/s ln(2/x) g2),  s = mu ln(2/x).
// The terms fall at least like 1/(k!)^2; at x = 2 fifteen reach the double rounding unit.
MATERN_FN inline void bessel_k_series(const MaternNu &n, double x, double &k0, double &k1) {
    const double lg = -log(0.5 * x);
    const double s = n.mu * lg;
    const double e = exp(s), ei = 1.0 / e;
    double f = n.fac * (0.5 * (e + ei) * n.g1 + sinh_ratio(s, e, ei) * lg * n.g2);
    const double p0 = e * n.ip, q0 = ei * n.iq;
    const double y = 0.25 * x * x;
    double p = p0, q = q0, yk = 1.0, s0 = f, s1 = p;
    for (int k = 1; k < MaternNu::KS; ++k) {
        const double dk = (double)k;
        f = (dk * f + p + q) * n.r2[k];
        p = p0 * n.rm[k];
        q = q0 * n.rp[k];
        yk *= y;
        const double c = yk * n.rf[k];
        const double t0 = c * f, t1 = c * (p - dk * f);
        s0 += t0;
        s1 += t1;
        if (fabs(t0) < 1e-17 * fabs(s0) && fabs(t1) < 1e-17 * fabs(s1)) break;
    }
    k0 = s0;
    k1 = s1 * (2.0 / x);
}

// e^x K_mu(x), e^x K_{mu+1}(x) for |mu| <= 1/2, x > 2.  U_k satisfies
//   U_{k-1} = 2(k+x) U_k - a_k U_{k+1},  a_k = (k+1/2)^2 - mu^2,
// taken backward from U_{K+1} = 0, U_K = 1 (at most 2^82 83! / 2, far from overflow), with the sum
// S = sum C_k U_k alongside, C_k / C_{k-1} = a_{k-1} / k; and then
// e^x K_mu = sqrt(pi / 2x) / (S / U_0),  K_{mu+1} / K_mu = (mu + 1/2 + x + (mu^2 - 1/4) U_1 / U_0) / x.
// K = 6 + 150/x terms keep the truncation below the rounding unit for every x > 2.
MATERN_FN inline void bessel_k_ratio(const MaternNu &n, double x, double &k0, double &k1) {
    const int K = 6 + (int)ceil(150.0 / x);
    double u1 = 0.0, u0 = 1.0, S = 0.0;                  // U_{k+1}, U_k
    double bk = 2.0 * (K + x);
    for (int k = K; k >= 1; --k) {
        S += n.c[k] * u0;
        const double u = bk * u0 - n.a[k] * u1;
        u1 = u0;
        u0 = u;
        bk -= 2.0;
    }
    S += u0;                                             // C_0 = 1
    k0 = sqrt(3.141592653589793 / (2.0 * x)) / (S / u0);
    k1 = k0 * (n.mu + 0.5 + x + (n.mu * n.mu - 0.25) * (u1 / u0)) / x;
}

// 2^(1-nu)/Gamma(nu) x^nu K_nu(x), the Matern correlation of Eq. 2 at x = h/a >= 0 (1 at 0).
// Below x <= 2 with nu ln(2/x) > 600 the value is 1 to far below the rounding unit (the
// deviation is O(x^2) for nu > 1 and O(x^(2 nu)) otherwise), and K_nu would overflow; above
// x = 1450, x^nu e^-x underflows for every nu <= 16.
MATERN_FN inline double matern_corr(const MaternNu &c, double x) {
    if (x == 0.0) return 1.0;
    if (x > 1450.0) return 0.0;
    const bool small = x <= 2.0;
    if (small && c.nu * log(2.0 / x) > 600.0) return 1.0;
    double k0, k1;
    if (small) bessel_k_series(c, x, k0, k1);
    else bessel_k_ratio(c, x, k0, k1);
    double kn = k0;
    if (c.m > 0) {
        for (int j = 1; j < c.m; ++j) {
            const double k2 = k0 + (2.0 * (c.mu + j) / x) * k1;
            k0 = k1;
            k1 = k2;
        }
        kn = k1;
    }
    if (small) return c.pre * (pow(x, c.nu) * kn);
    const double h = exp(-0.5 * x);               // e^-x in two halves: x^nu e^-x/2 stays finite
    return c.pre * ((pow(x, c.nu) * h) * (kn * h));
}

// x = h / a of two points, h = |s_i - s_j|: bit for bit the plain IEEE evaluation (every operation
// rounded, no contraction), with the square root and the quotient in integer arithmetic where their
// arguments are in range.
struct Range {
    double a;
    fx::Divisor d, three;
    int fast;            // a lies in [1e-100, 1e100]
};
__device__ __forceinline__ double scaled_distance(double dx, double dy, const Range &g, fx::Num &x) {
    const double s = __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
    if (g.fast && s > 1e-150 && s < 1e150) {
        x = fx::div_rn(fx::sqrt_rn(s), g.d);
        return fx::value(x);
    }
    return __ddiv_rn(__dsqrt_rn(s), g.a);
}

// One CTA row (blockIdx.y) per tile; a CTA takes whole columns of it, its threads the rows (several
// columns at once for a tile of less than 256 rows), so a thread's own point stays in registers and
// consecutive threads write consecutive rows.  Every operation is rounded on its own, so h and
// x = h/a are bit-identical to a plain IEEE evaluation, and only e^-x may differ (by its last bit)
// from another library.  Bound by the FP64 pipe and the integer units together: 8 FP64 and about 180
// integer operations an element.  The matrix of order 32768, nu = 3/2, takes 13.8 ms; with the FP64
// library's square root, division and exponential (42 FP64 operations) it took 43.7 ms.
template <int NU2>
__global__ void __launch_bounds__(256)
k_matern(double *A, int64_t n, int b, const double *__restrict__ pts, double sigma2, const __grid_constant__ Range g,
         const __grid_constant__ MaternNu general, double nugget) {
    __shared__ uint64_t table[NU2 ? fx::EXP_TABLE : 1];
    __shared__ __align__(16) unsigned char cbuf[NU2 ? 1 : sizeof(MaternNu)];    // lanes read its tables at their own k
    const MaternNu &cn = *reinterpret_cast<const MaternNu *>(cbuf);
    if (NU2 == 0) {
        for (int i = threadIdx.x; i < (int)(sizeof(MaternNu) / 4); i += 256)
            reinterpret_cast<uint32_t *>(cbuf)[i] = reinterpret_cast<const uint32_t *>(&general)[i];
    }
    if (NU2)
        for (int i = threadIdx.x; i < fx::EXP_TABLE; i += 256) table[i] = fx::exp_entry(i);
    const int t = blockIdx.y;
    // tile (i, j) from the packed index t = i(i+1)/2 + j
    int i = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while (i * (i + 1) / 2 > t) --i;
    while ((i + 1) * (i + 2) / 2 <= t) ++i;
    const int j = t - i * (i + 1) / 2;
    double *T = A + (int64_t)t * b * b;
    const int rows = b < 256 ? b : 256, cpp = 256 / rows;            // rows and columns of a pass
    const int tr = threadIdx.x % rows, tc = threadIdx.x / rows;
    __syncthreads();
    if (tc >= cpp) return;
    for (int r = tr; r < b; r += rows) {
        const int64_t gi = (int64_t)i * b + r;
        const double xi = gi < n ? pts[2 * gi] : 0.0, yi = gi < n ? pts[2 * gi + 1] : 0.0;
        for (int c = blockIdx.x * cpp + tc; c < b; c += gridDim.x * cpp) {
            const int64_t gj = (int64_t)j * b + c;
            double v;
            if (gi >= n || gj >= n) {
                v = (gi == gj) ? 1.0 : 0.0;
            } else {
                fx::Num xn{0, 0};
                const double x = scaled_distance(__dsub_rn(xi, pts[2 * gj]), __dsub_rn(yi, pts[2 * gj + 1]), g, xn);
                double f;
                if constexpr (NU2 == 0) {
                    f = matern_corr(cn, x);
                } else {
                    const double ex = (xn.m && x < 700.0) ? fx::exp_neg(xn, table) : exp(-x);
                    if constexpr (NU2 == 1) f = ex;
                    else if constexpr (NU2 == 3) f = __dmul_rn(__dadd_rn(1.0, x), ex);
                    else {
                        const double xx = __dmul_rn(x, x);
                        double third;
                        if (xx > 1e-250 && xx < 1e250) {
                            const uint64_t w = fx::bits(xx);
                            third = fx::value(fx::div_rn({(w & 0xFFFFFFFFFFFFFull) | (1ull << 52), (int)(w >> 52) - 1075}, g.three));
                        } else {
                            third = __ddiv_rn(xx, 3.0);
                        }
                        f = __dmul_rn(__dadd_rn(__dadd_rn(1.0, x), third), ex);
                    }
                }
                v = sigma2 == 1.0 ? f : __dmul_rn(sigma2, f);
                if (gi == gj) v = __dadd_rn(v, nugget);
            }
            T[(int64_t)c * b + r] = v;
        }
    }
}

// Sum of squares of tile t0 + blockIdx.x / 8 (global packed index; the tile itself at
// A + (blockIdx.x / 8) b^2), padding excluded: a cluster of eight CTAs per tile, each the columns of
// an eighth of it, whose sums meet in the cluster's first CTA in a fixed order.  Bound by the FP64
// pipe (one multiply-add an element, 1.0 ms for a matrix of order 32768) and then by the bytes
// (0.63 ms); one CTA per tile with 8-byte loads and a division for every element's row and column
// took 8.8 ms (136 tiles of 2048 on 152 SMs).
constexpr int SUMSQ_CLUSTER = 8;
__global__ void __cluster_dims__(SUMSQ_CLUSTER, 1, 1) __launch_bounds__(256)
k_tile_sumsq(const double *A, int b, int64_t n, double *out, int t0) {
    __shared__ double red[8];
    __shared__ double part;
    const int rank = (int)blockIdx.x % SUMSQ_CLUSTER, lt = (int)blockIdx.x / SUMSQ_CLUSTER, t = t0 + lt;
    int i = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while ((int64_t)i * (i + 1) / 2 > t) --i;
    while ((int64_t)(i + 1) * (i + 2) / 2 <= t) ++i;
    const int j = t - (int)((int64_t)i * (i + 1) / 2);
    const double *T = A + (int64_t)lt * b * b;
    const int nvr = (int)min((int64_t)b, n - (int64_t)i * b), nvc = (int)min((int64_t)b, n - (int64_t)j * b);
    const int c0 = rank * (b / SUMSQ_CLUSTER), c1 = min(nvc, c0 + b / SUMSQ_CLUSTER);
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    if (nvr == b && ((uintptr_t)A & 15) == 0) {          // whole columns: one run of 16-byte loads
        const double2 *p = reinterpret_cast<const double2 *>(T + (int64_t)c0 * b);
        const int64_t m = c1 > c0 ? (int64_t)(c1 - c0) * b / 2 : 0;
        int64_t e = threadIdx.x;
        for (; e + 768 < m; e += 1024) {
            const double2 u = p[e], v = p[e + 256], w = p[e + 512], x = p[e + 768];
            s0 = fma(u.x, u.x, s0);
            s1 = fma(u.y, u.y, s1);
            s2 = fma(v.x, v.x, s2);
            s3 = fma(v.y, v.y, s3);
            s0 = fma(w.x, w.x, s0);
            s1 = fma(w.y, w.y, s1);
            s2 = fma(x.x, x.x, s2);
            s3 = fma(x.y, x.y, s3);
        }
        for (; e < m; e += 256) {
            const double2 u = p[e];
            s0 = fma(u.x, u.x, s0);
            s1 = fma(u.y, u.y, s1);
        }
    } else {
        for (int c = c0; c < c1; ++c)
            for (int r = threadIdx.x; r < nvr; r += 256) {
                const double v = T[(int64_t)c * b + r];
                s0 = fma(v, v, s0);
            }
    }
    double s = (s0 + s1) + (s2 + s3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += red[w];
        part = v;
    }
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    cl.sync();
    if (rank == 0 && threadIdx.x == 0) {
        double v = 0.0;
        for (int q = 0; q < SUMSQ_CLUSTER; ++q) v += *cl.map_shared_rank(&part, q);
        out[t] = v;
    }
    cl.sync();                                           // `part` stays until it has been read
}

void launch_matern(double *A, int64_t n, int b, int nt, const double *pts, double sigma2, double a,
                   int nu2, double nu, double nugget, cudaStream_t s) {
    const int T = nt * (nt + 1) / 2;
    // 16 elements a thread (a CTA fills a table of 1024 entries first), 64 CTAs a tile at most; few tiles
    // take as many CTAs as fill the SMs with eight each, down to a column a CTA (nu = 0.8, 15 tiles of 128:
    // 835 us with four CTAs a tile, 281 us; nu = 3/2, 6 tiles of 256: 50 and 40 us)
    int gx = (int)((int64_t)b * b / 4096);
    gx = gx < 1 ? 1 : gx > 64 ? 64 : gx;
    const int fill = (8 * NSM + T - 1) / T, columns = b < 256 ? b / (256 / b) : b;
    gx = std::max(gx, std::min(fill, columns));
    Range g{};
    g.a = a;
    g.fast = a > 1e-100 && a < 1e100;
    if (g.fast) g.d = fx::make_divisor(a);
    g.three = fx::make_divisor(3.0);
    const dim3 grid(gx, T);
    if (nu2 == 1) k_matern<1><<<grid, 256, 0, s>>>(A, n, b, pts, sigma2, g, MaternNu{}, nugget);
    else if (nu2 == 3) k_matern<3><<<grid, 256, 0, s>>>(A, n, b, pts, sigma2, g, MaternNu{}, nugget);
    else if (nu2 == 5) k_matern<5><<<grid, 256, 0, s>>>(A, n, b, pts, sigma2, g, MaternNu{}, nugget);
    else k_matern<0><<<grid, 256, 0, s>>>(A, n, b, pts, sigma2, g, matern_nu(nu), nugget);
}

void launch_tile_sumsq(const double *A, int nt, int b, int64_t n, double *out, cudaStream_t s) {
    const int T = nt * (nt + 1) / 2;
    k_tile_sumsq<<<T * SUMSQ_CLUSTER, 256, 0, s>>>(A, b, n, out, 0);
}
void launch_tile_sumsq_range(const double *A_first, int t0, int count, int b, int64_t n, double *out, cudaStream_t s) {
    if (count > 0) k_tile_sumsq<<<count * SUMSQ_CLUSTER, 256, 0, s>>>(A_first, b, n, out, t0);
}

}  // namespace tc
