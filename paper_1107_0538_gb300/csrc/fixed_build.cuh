// Builds a handle's fixed-point matrix copy (fixed.cuh) from its SELL-32 copy,
// once at creation: the row exponents, the exponent of the largest entry, then
// the integers.  One warp per slice, lane per row; three passes over the
// matrix at most.
#pragma once

#include "fixed.cuh"

namespace gbcg {

// c_i from the diagonal.  flags: set when the matrix is not eligible.
__global__ void __launch_bounds__(256) fixed_scale_kernel(SellMatrix M, int8_t *c, unsigned int *flags, unsigned int *maxc) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (t >= M.nslices) return;
    const int row = t * 32 + lane;
    if (row >= M.n) return;
    const long long a = M.ptr[t];
    const int w = (int)((M.ptr[t + 1] - a) >> 5);
    double d = 0.0;
    int m = 0;   // products that can be other than zero: the slice's width also counts padding
    for (int k = 0; k < w; ++k) {
        const long long i = a + 32LL * k + lane;
        const int col = M.cols16 ? row + M.cols16[i] : M.cols32[i];
        const double v = M.vals[i];
        if (col == row) d += v;
        m += v != 0.0;
    }
    const int e = (int)((unsigned long long)__double_as_longlong(d) >> 52);   // with the sign bit
    const int ci = (e - 1023 + 1) >> 1;
    if (m > kFixedMaxWidth || e == 0 || e >= 2047 || ci > kFixedMaxC || ci < -kFixedMaxC) {
        atomicOr(flags, 1u);
        c[row] = 0;
        return;
    }
    c[row] = (int8_t)ci;
    atomicMax(maxc, (unsigned int)(128 + ci));       // maxc[0] - 128 = max c_i,
    atomicMax(maxc + 1, (unsigned int)(128 - ci));   // 128 - maxc[1] = min c_i
}

// The smallest x (plus kFixedExpOffset) with every |a_ij| 2^(-c_i - c_j) < 2^x
// and every row's sum of them < 2^(x + 3); entries that are not finite raise
// the flag.
constexpr int kFixedExpOffset = 4096;
__global__ void __launch_bounds__(256)
    fixed_max_kernel(SellMatrix M, const int8_t *c, unsigned int *flags, unsigned int *maxexp) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (t >= M.nslices) return;
    const int row = t * 32 + lane;
    int x = 0;
    if (row < M.n) {
        const long long a = M.ptr[t];
        const int w = (int)((M.ptr[t + 1] - a) >> 5);
        const int cr = c[row];
        double sum = 0.0;
        for (int k = 0; k < w; ++k) {
            const long long i = a + 32LL * k + lane;
            const int col = M.cols16 ? row + M.cols16[i] : M.cols32[i];
            const double v = M.vals[i];
            const int e = (__double2hiint(v) >> 20) & 0x7ff;
            if (e == 0x7ff) atomicOr(flags, 1u);
            if (e != 0) {
                x = max(x, e - 1022 - cr - c[col] + kFixedExpOffset);
                sum += ldexp(fabs(v), -cr - c[col]);
            }
        }
        if (sum > 0.0) x = max(x, ((__double2hiint(sum) >> 20) & 0x7ff) - 1022 - 3 + kFixedExpOffset);
    }
    const unsigned int m = __reduce_max_sync(0xffffffffu, (unsigned int)x);
    if (lane == 0 && m) atomicMax(maxexp, m);
}

__global__ void __launch_bounds__(256)
    fixed_build_kernel(SellMatrix M, const int8_t *c, int u, int2 *vals) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (t >= M.nslices) return;
    const int row = t * 32 + lane;
    const long long a = M.ptr[t];
    const int w = (int)((M.ptr[t + 1] - a) >> 5);
    for (int k = 0; k < w; ++k) {
        const long long i = a + 32LL * k + lane;
        int2 v = make_int2(0, 0);
        if (row < M.n) {
            const int col = M.cols16 ? row + M.cols16[i] : M.cols32[i];
            v = fixed_split(fixed_of((unsigned long long)__double_as_longlong(M.vals[i]), u - c[row] - c[col]),
                            kFixedLoBits);
        }
        vals[i] = v;
    }
}

}  // namespace gbcg
