// The FP64 building blocks of the SELL-32 solve kernels (1024 threads a CTA,
// one per SM), shared by the CG solves and the flexible-CG iteration: row
// sums of a slice, and fixed-order sums over the CTA and over the grid.
#pragma once

#include "cg_device.cuh"
#include "fixed.cuh"
#include "sell.cuh"

namespace gbcg {

constexpr int kSellSolveThreads = 1024;
constexpr int kSellUnrollMem = 18;   // loads in flight per row where rows are not held in registers

// a / b or its neighbour in the last place, for the scalars of an iteration: Newton's step
// for the reciprocal from a single-precision seed y (error 2^-22), folded into
// the quotient, and one correction with the exact remainder (Markstein, "Computation
// of elementary functions on the IBM RISC System/6000", 1990): five FP64
// operations of 64 clocks, where a call of the division takes 580.
__device__ __forceinline__ double scalar_quotient(double a, double b) {
    const unsigned int ha = (unsigned int)__double2hiint(a), hb = (unsigned int)__double2hiint(b);
    const int ea = (int)(ha >> 20) & 0x7ff, eb = (int)(hb >> 20) & 0x7ff;
    if (ea < 64 || ea > 1982 || eb < 64 || eb > 1982 || abs(ea - eb) > 900) return a / b;
    // b = 2^(eb - 1023) m, m in [1, 2) with b's sign
    const double m = __hiloint2double((int)((hb & 0x800fffffu) | 0x3ff00000u), __double2loint(b));
    const unsigned int mf = ((hb & 0xfffffu) << 3) | ((unsigned int)__double2loint(b) >> 29);
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__uint_as_float(0x3f800000u | mf)));
    const unsigned int yb = __float_as_uint(yf);   // in (1/2, 1]
    const double y = __hiloint2double((int)(((yb >> 3) + ((1023u - 127u) << 20)) | (hb & 0x80000000u)), (int)(yb << 29));
    const double q0 = a * y;
    const double e = fma(-m, y, 1.0);
    const double q1 = fma(q0, e, q0);
    const double q = fma(fma(-m, q1, a), y, q1);
    // times 2^(1023 - eb): the exponents stay inside the normal range
    return __hiloint2double(__double2hiint(q) + ((1023 - eb) << 20), __double2loint(q));
}

// Sums over the CTA in a fixed order with the FP64 work spread over the four
// SM sub-partitions (warp w issues on sub-partition w mod 4; one warp-wide
// FP64 add occupies a sub-partition's FP64 pipe for ~64 cycles, so the number
// of adds on the busiest sub-partition is the cost).  Quarter g of 32
// partials per lane is added by warp g and folded by a butterfly; lane j of
// warp 0 then adds the four quarter sums of value j.  Thread 0 ends with the
// totals, the same bits in every CTA and every run.
//
// Two values share one butterfly: lanes 0-15 fold value 0 and lanes 16-31
// value 1 after the first exchange.
template <int NV>
__device__ __forceinline__ void fold_quarter(double (&t)[NV], double *quarter, int g) {
    const int lane = threadIdx.x & 31;
    if constexpr (NV == 2) {
        const bool lo = lane < 16;
        const double keep = lo ? t[0] : t[1];
        double u = keep + __shfl_xor_sync(0xffffffffu, lo ? t[1] : t[0], 16);
#pragma unroll
        for (int m = 8; m >= 1; m >>= 1) u += __shfl_xor_sync(0xffffffffu, u, m);
        if (lane == 0) quarter[g] = u;
        if (lane == 16) quarter[4 + g] = u;
    } else {
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            const double u = warp_sum(t[j]);
            if (lane == 0) quarter[4 * j + g] = u;
        }
    }
}

// Thread 0 (and every lane of warp 0) gets the totals of the four quarters.
template <int NV>
__device__ __forceinline__ void add_quarters(double (&v)[NV], const double *quarter) {
    const int lane = threadIdx.x & 31;
    double t = 0.0;
    if (lane < NV) {
        const double *q = quarter + 4 * lane;
        t = (q[0] + q[1]) + (q[2] + q[3]);
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) v[j] = __shfl_sync(0xffffffffu, t, j);
}

//
// With wmax (kMaxSlots words of shared memory) the largest mx of the CTA is
// formed on the way, on warps the sums leave idle, in wmax[32].
constexpr int kMaxSlots = 34;
template <int NV>
__device__ __forceinline__ void block_sum_1k(double (&v)[NV], double *red, double *quarter, unsigned int *wmax = nullptr,
                                             unsigned int mx = 0) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (wmax) {
        const unsigned int m = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) wmax[w] = m;
    }
#pragma unroll
    for (int j = 0; j < NV; ++j) red[j * kSellSolveThreads + threadIdx.x] = v[j];
    __syncthreads();
    if (w < 4) {
        double t[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            // 8 partials per lane, added as a tree (depth 3, not a chain of 7)
            const double *src = red + j * kSellSolveThreads + 32 * w + lane;
            static_assert(kSellSolveThreads / 128 == 8, "8 partials per lane");
            t[j] = ((src[0] + src[128]) + (src[256] + src[384])) + ((src[512] + src[640]) + (src[768] + src[896]));
        }
        fold_quarter<NV>(t, quarter, w);
    } else if (wmax && w == 4) {
        const unsigned int m = __reduce_max_sync(0xffffffffu, wmax[lane]);
        if (lane == 0) wmax[32] = m;
    }
    __syncthreads();
    if (w == 0) add_quarters<NV>(v, quarter);
}

// The CTA's maximum travels in the last slot of its partial-sum record.
__device__ __forceinline__ void publish_max(const Params &P, int set, unsigned int mx) {
    if (threadIdx.x == 0)
        reinterpret_cast<long long *>(P.partials)[((size_t)set * gridDim.x + blockIdx.x) * kRedSlots + kRedSlots - 1] = mx;
}

// Largest maximum of every CTA's record (one warp; all its lanes get it).
__device__ __forceinline__ unsigned int grid_max(const Params &P, int set) {
    const int G = (int)gridDim.x;
    const long long *src = reinterpret_cast<const long long *>(P.partials) + (size_t)set * G * kRedSlots + kRedSlots - 1;
    unsigned int m = 0;
    for (int c = threadIdx.x & 31; c < G; c += 32) m = max(m, (unsigned int)__ldcg(src + (size_t)c * kRedSlots));
    return __reduce_max_sync(0xffffffffu, m);
}

// Grid totals of the partials of barrier set `set`: warp g < 4 adds the
// partials of CTAs g*32 + lane + 128 u, then as above.  Every CTA computes
// the same bits.
template <int NV>
__device__ __forceinline__ void grid_totals_1k(const Params &P, int set, double (&out)[NV], double *quarter,
                                               unsigned int *wmax = nullptr) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int G = (int)gridDim.x;
    if (w < 4) {
        const double *src = P.partials + (size_t)set * G * kRedSlots;
        double t[NV];
        const int m0 = 32 * w + lane;
#pragma unroll
        for (int j = 0; j < NV; ++j) t[j] = m0 < G ? __ldcg(src + (size_t)m0 * kRedSlots + j) : 0.0;
        for (int m = m0 + 128; m - lane < G; m += 128) {
#pragma unroll
            for (int j = 0; j < NV; ++j) t[j] += m < G ? __ldcg(src + (size_t)m * kRedSlots + j) : 0.0;
        }
        fold_quarter<NV>(t, quarter, w);
    } else if (wmax && w == 4) {
        const unsigned int m = grid_max(P, set);
        if (lane == 0) wmax[33] = m;   // with wmax: the largest maximum, for thread 0
    }
    __syncthreads();
    if (w == 0) add_quarters<NV>(out, quarter);
}

// init + row sum of lane's row in slice t (all 32 lanes of the warp call it),
// one accumulator: seven warps per SM sub-partition keep its FP64 pipe busy,
// so the chain's latency is hidden, and starting from init (beta q in the
// iteration) saves the separate add of the recurrence.  x is written by this
// kernel between grid barriers, so its loads are plain coherent loads
// (L1-cached: the acquire fence of every grid barrier drops stale L1 lines),
// never the read-only path; the matrix goes through L2 only, leaving L1 to
// the gathered window of x.
// Entries k0 <= k < k1 of the slice (k1 < 0: to the slice width), in
// batches of U entries (all loads of a batch in flight before its FMAs),
// then of kSellUnroll, then one at a time.
// sell_slice_sum_at takes the slice's first entry a and its width wt (a
// caller that keeps them saves the two dependent loads of M.ptr per call).
template <int U = kSellUnroll>
__device__ __forceinline__ double sell_slice_sum_at(const SellMatrix &M, int t, long long a, int wt, const double *x,
                                                    double init, int k0 = 0, int k1 = -1) {
    const int lane = threadIdx.x & 31;
    const bool st = M.stream != 0;
    const int w = k1 >= 0 ? k1 : wt;
    const int row = t * 32 + lane;
    const double *vv = M.vals + a + lane;
    double s = init;
    int k = k0;
    if (M.cols16) {
        const int16_t *cc = M.cols16 + a + lane;
        if constexpr (U != kSellUnroll) {
            for (; k + U <= w; k += U) {
                double vr[U], xr[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    vr[u] = mload(vv + (k + u) * 32, st);
                    xr[u] = __ldca(x + bchk(row + (int)mload(cc + (k + u) * 32, st), M.n));
                }
#pragma unroll
                for (int u = 0; u < U; ++u) s = fma(vr[u], xr[u], s);
            }
        }
        for (; k + kSellUnroll <= w; k += kSellUnroll) {
            double vr[kSellUnroll], xr[kSellUnroll];
#pragma unroll
            for (int u = 0; u < kSellUnroll; ++u) {
                vr[u] = mload(vv + (k + u) * 32, st);
                xr[u] = __ldca(x + bchk(row + (int)mload(cc + (k + u) * 32, st), M.n));
            }
#pragma unroll
            for (int u = 0; u < kSellUnroll; ++u) s = fma(vr[u], xr[u], s);
        }
        for (; k < w; ++k) s = fma(mload(vv + k * 32, st), __ldca(x + bchk(row + (int)mload(cc + k * 32, st), M.n)), s);
    } else {
        const int32_t *cc = M.cols32 + a + lane;
        if constexpr (U != kSellUnroll) {
            for (; k + U <= w; k += U) {
                double vr[U], xr[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    vr[u] = mload(vv + (k + u) * 32, st);
                    xr[u] = __ldca(x + bchk(mload(cc + (k + u) * 32, st), M.n));
                }
#pragma unroll
                for (int u = 0; u < U; ++u) s = fma(vr[u], xr[u], s);
            }
        }
        for (; k + kSellUnroll <= w; k += kSellUnroll) {
            double vr[kSellUnroll], xr[kSellUnroll];
#pragma unroll
            for (int u = 0; u < kSellUnroll; ++u) {
                vr[u] = mload(vv + (k + u) * 32, st);
                xr[u] = __ldca(x + bchk(mload(cc + (k + u) * 32, st), M.n));
            }
#pragma unroll
            for (int u = 0; u < kSellUnroll; ++u) s = fma(vr[u], xr[u], s);
        }
        for (; k < w; ++k) s = fma(mload(vv + k * 32, st), __ldca(x + bchk(mload(cc + k * 32, st), M.n)), s);
    }
    return s;
}

template <int U = kSellUnroll>
__device__ __forceinline__ double sell_slice_sum(const SellMatrix &M, int t, const double *x, double init,
                                                 int k0 = 0, int k1 = -1) {
    const long long a = M.ptr[t];
    return sell_slice_sum_at<U>(M, t, a, (int)((M.ptr[t + 1] - a) >> 5), x, init, k0, k1);
}

}  // namespace gbcg
