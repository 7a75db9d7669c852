// SpMV in the SELL-32 layout, read straight from global memory (sm_103a).
//
// Slice t holds rows 32t .. 32t+31 padded to the longest of them (w_t
// entries); entry k of lane l sits at offset slice_ptr[t] + 32 k + l, so the
// warp that owns a slice reads 32 consecutive values, 32 consecutive
// columns and, for a stencil (the k-th neighbour of consecutive rows is at
// a constant offset), 32 consecutive entries of x per step: every load is
// coalesced, nothing is staged in shared memory, and any number of warps
// can run per SM.  Columns are 16-bit offsets from the row (cols16) when
// every |col - row| < 2^15, else 32-bit column indices (cols32).  Padded
// entries have value 0 and point at the row itself.
//
// Exactly one FMA per stored entry (plus padding, below 1% for Q1 boxes);
// the summation order differs from the tiled kernels only in association.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "check.cuh"

namespace gbcg {

struct SellMatrix {
    int32_t n;
    int32_t nslices;
    int32_t stream;                        // 1: matrix loads marked evict-first (matrix larger than L2)
    const long long *__restrict__ ptr;     // nslices + 1 entry offsets (multiples of 32)
    const double *__restrict__ vals;       // padded entries
    const int16_t *__restrict__ cols16;    // col - row, or nullptr
    const int32_t *__restrict__ cols32;    // col, when cols16 is nullptr
    const int32_t *__restrict__ split;     // per slice: width of the block of entries in the CTA's own
                                           // rows (slice solve kernel layout), or nullptr
};

constexpr int kSellThreads = 256;
// Four CTAs an SM, 64 registers a thread: with eight (32 registers) the loads
// of a batch cannot be in flight together and a system of one or two slices per
// warp waits for them one after the other.  Eight against four, us per call,
// three matrices in turn: up to 32^3 10.25 / 6.16, 50^3 20.5 / 14.4, 57^3 20.5 /
// 17.0, 72^3 28.7 / 26.5, 80^3 and 100^3 32.9 and 57.3 either way.  Batches of 14
// and 27 with three, two or one CTAs were slower from 40^3 on (100^3 61 to 83).
// Half as many warps only pay with a row's rest in one batch too: entry by
// entry, short rows fell behind the eight CTAs.  Eight / four, entry by entry / four,
// one batch, us per call in a row: 3 entries a row, 1.2M rows 14.5 / 20.7 / 14.8 (2.4M
// 23.1 / 36.6 / 25.5); 5-point 2000^2 49.5 / 57.8 / 51.6; 7-point 90^3 16.8 / 20.5 / 16.6;
// 21 entries, 1.2M rows 55.9 / 58.2 / 53.5; Q1 72^3 29.0 / 26.2 / 24.9, 100^3 59.5 / 57.5 /
// 55.6.  (Reading the next slice's place ahead: 2400000 x 3 24.9, but Q1 100^3 56.4.)
constexpr int kSellBlocksPerSm = 4;
constexpr int kSellUnroll = 9;

// Matrix loads: streaming (evict-first, read once per SpMV) when the matrix
// does not fit L2, plain (kept in L2 across SpMVs) when it does.
template <class T>
__device__ __forceinline__ T mload(const T *p, bool stream) {
    return stream ? __ldcs(p) : __ldcg(p);
}

// Entries k .. k + N - 1 of lane's row, all their loads in flight before the
// FMAs: even ones into s0, odd ones into s1, or (TAIL) all into s0, in order.
template <int N, bool TAIL, class Col>
__device__ __forceinline__ void sell_batch(const SellMatrix &M, const double *vv, const Col *cc, int base, int k,
                                           const double *__restrict__ x, double &s0, double &s1) {
    const bool st = M.stream != 0;
    double vr[N], xr[N];
#pragma unroll
    for (int u = 0; u < N; ++u) {
        vr[u] = mload(vv + (k + u) * 32, st);
        xr[u] = __ldg(x + bchk(base + (int)mload(cc + (k + u) * 32, st), M.n));
    }
#pragma unroll
    for (int u = 0; u < N; ++u) {
        if (!TAIL && (u & 1)) s1 = fma(vr[u], xr[u], s1);
        else s0 = fma(vr[u], xr[u], s0);
    }
}

// Lane's row of a slice of width w in batches of kSellUnroll, the rest in one
// batch of its size (the branches are the warp's).
template <class Col>
__device__ __forceinline__ double sell_row(const SellMatrix &M, const double *vv, const Col *cc, int base, int w,
                                           const double *__restrict__ x) {
    double s0 = 0.0, s1 = 0.0;
    int k = 0;
    for (; k + kSellUnroll <= w; k += kSellUnroll) sell_batch<kSellUnroll, false>(M, vv, cc, base, k, x, s0, s1);
    static_assert(kSellUnroll == 9, "cases below");
    switch (w - k) {
        case 8: sell_batch<8, true>(M, vv, cc, base, k, x, s0, s1); break;
        case 7: sell_batch<7, true>(M, vv, cc, base, k, x, s0, s1); break;
        case 6: sell_batch<6, true>(M, vv, cc, base, k, x, s0, s1); break;
        case 5: sell_batch<5, true>(M, vv, cc, base, k, x, s0, s1); break;
        case 4: sell_batch<4, true>(M, vv, cc, base, k, x, s0, s1); break;
        case 3: sell_batch<3, true>(M, vv, cc, base, k, x, s0, s1); break;
        case 2: sell_batch<2, true>(M, vv, cc, base, k, x, s0, s1); break;
        case 1: sell_batch<1, true>(M, vv, cc, base, k, x, s0, s1); break;
        default: break;
    }
    return s0 + s1;
}

// Row sums of the slices owned by this warp (grid-stride over slices):
// epi.row(i, sum) for every row i < n.
template <class Epi>
__device__ __forceinline__ void sell_rows(const SellMatrix &M, const double *__restrict__ x, Epi &epi) {
    const int lane = threadIdx.x & 31;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int t = warp; t < M.nslices; t += nwarps) {
        const long long a = M.ptr[t];
        const int w = (int)((M.ptr[t + 1] - a) >> 5);
        const int row = t * 32 + lane;
        const double sum = M.cols16 ? sell_row(M, M.vals + a + lane, M.cols16 + a + lane, row, w, x)
                                    : sell_row(M, M.vals + a + lane, M.cols32 + a + lane, 0, w, x);
        if (row < M.n) epi.row(row, sum, 0);
    }
}

}  // namespace gbcg
