// Arrays through the functions of fixed_exp.h, for test_fixed_exp.py: compiled as C++ on the host, or with
// nvcc for the device.  op 0: sqrt_rn(x); 1, 2: root and reciprocal of sqrt_recip_rn(x); 3: x / y by div_rn;
// 4: exp_neg(x).
#ifdef __CUDACC__
#define FIXED_FN __host__ __device__ __forceinline__
#else
#define FIXED_FN static inline
#endif
#include "fixed_exp.h"

using namespace tc::fx;

FIXED_FN Num number(double x) { return {(bits(x) & 0xFFFFFFFFFFFFFull) | (1ull << 52), (int)(bits(x) >> 52) - 1075}; }
FIXED_FN double apply(int op, double x, double y, const uint64_t *table) {
    Num a, b;
    switch (op) {
        case 0: return value(sqrt_rn(x));
        case 1: sqrt_recip_rn(x, a, b); return value(a);
        case 2: sqrt_recip_rn(x, a, b); return value(b);
        case 3: return value(div_rn(number(x), make_divisor(y)));
        default: return exp_neg(number(x), table);
    }
}

#ifdef __CUDACC__
__global__ void k_apply(int op, const double *x, const double *y, double *out, int n, const uint64_t *table) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = apply(op, x[i], y[i], table);
}
#endif

// x, y, out: n values, table: EXP_TABLE words; in host memory, or on the device when compiled by nvcc.
// Returns 0, or the CUDA error.
extern "C" int apply_all(int op, const double *x, const double *y, double *out, int n, const uint64_t *table) {
#ifdef __CUDACC__
    k_apply<<<(n + 255) / 256, 256>>>(op, x, y, out, n, table);
    const cudaError_t e = cudaGetLastError();
    return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
#else
    for (int i = 0; i < n; ++i) out[i] = apply(op, x[i], y[i], table);
    return 0;
#endif
}
extern "C" void fill_table(uint64_t *table) {
    for (int i = 0; i < EXP_TABLE; ++i) table[i] = exp_entry(i);
}
