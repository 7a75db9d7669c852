// Builds a handle's slices with common offsets (ring.cuh) from its SELL-32
// copy, once at creation, on the device: the offsets of every slice, then, with
// the slices' places known, the values.  One warp per slice.
#pragma once

#include <cuda_bf16.h>

#include "fixed.cuh"
#include "ring.cuh"

namespace gbcg {

constexpr int kRingMaxWidth = 32;   // offsets per slice at most (one per lane)

// The sorted union of the offsets of slice t's rows (offset of lane k in lane
// k) and its size; kRingMaxWidth + 1 when there are more.  An entry that is
// exactly the SELL padding (value zero at the row itself) adds nothing unless
// the row stores its diagonal.  `dup` is raised when a row has two entries in
// one column.
__device__ __forceinline__ int ring_offsets(const SellMatrix &M, int t, int *off_of_lane, bool &dup) {
    const int lane = threadIdx.x & 31, row = t * 32 + lane;
    const long long a = M.ptr[t];
    const int w = (int)((M.ptr[t + 1] - a) >> 5);
    int last = INT32_MIN, n = 0;
    *off_of_lane = 0;
    for (;;) {
        int best = INT32_MAX, hits = 0;
        if (row < M.n)
            for (int k = 0; k < w; ++k) {
                const long long i = a + 32LL * k + lane;
                const int o = M.cols16 ? (int)M.cols16[i] : M.cols32[i] - row;
                if (o <= last || o > best || (o == 0 && M.vals[i] == 0.0)) continue;
                hits = o == best ? hits + 1 : 1;
                best = o;
            }
        const int next = __reduce_min_sync(0xffffffffu, best);
        if (next == INT32_MAX) break;
        if (best == next && hits > 1) dup = true;
        if (n == kRingMaxWidth) return kRingMaxWidth + 1;
        if (lane == n) *off_of_lane = next;
        last = next;
        ++n;
    }
    return n;
}

// width[t], and flags: [0] not eligible, [1] largest |offset|.
__global__ void __launch_bounds__(256) ring_count_kernel(SellMatrix M, int32_t *width, unsigned int *flags) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (t >= M.nslices) return;
    int off = 0;
    bool dup = false;
    const int n = ring_offsets(M, t, &off, dup);
    if (lane == 0) width[t] = n;
    const unsigned int mx = __reduce_max_sync(0xffffffffu, lane < n ? (unsigned int)abs(off) : 0u);
    if (n > kRingMaxWidth || __any_sync(0xffffffffu, dup)) atomicOr(flags, 1u);
    if (lane == 0) atomicMax(flags + 1, mx);
}

// Values of the slices: fixed-point integers (VT = int2), or the off-diagonals
// rounded to nearest-even in VT (float, BF16 bits) and zero on the diagonal,
// where every zero is -0: +0 marks an offset that the row does not have.
template <class VT>
__device__ __forceinline__ VT ring_convert(double v, int row, int off, const int8_t *c, int u);
template <>
__device__ __forceinline__ int2 ring_convert<int2>(double v, int row, int off, const int8_t *c, int u) {
    return fixed_split(fixed_of((unsigned long long)__double_as_longlong(v), u - c[row] - c[row + off]), kFixedLoBits);
}
template <>
__device__ __forceinline__ float ring_convert<float>(double v, int, int off, const int8_t *, int) {
    const float f = off == 0 ? 0.0f : __double2float_rn(v);
    return f == 0.0f ? -0.0f : f;
}
template <>
__device__ __forceinline__ __nv_bfloat16 ring_convert<__nv_bfloat16>(double v, int, int off, const int8_t *, int) {
    const __nv_bfloat16 f = __double2bfloat16(off == 0 ? 0.0 : v);
    return __bfloat162float(f) == 0.0f ? __ushort_as_bfloat16(0x8000) : f;
}
__device__ __forceinline__ void ring_zero(int2 &v) { v = make_int2(0, 0); }
__device__ __forceinline__ void ring_zero(float &v) { v = 0.0f; }
__device__ __forceinline__ void ring_zero(__nv_bfloat16 &v) { v = __ushort_as_bfloat16(0); }

template <class VT>
__global__ void __launch_bounds__(256)
    ring_fill_kernel(SellMatrix M, const int2 *meta, unsigned char *blob, const int8_t *c, int u) {
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (t >= M.nslices) return;
    int off = 0;
    bool dup = false;
    const int n = ring_offsets(M, t, &off, dup), row = t * 32 + lane;
    const int2 me = meta[t];
    if (n != me.y) return;   // the count kernel saw the same slice
    unsigned char *dst = blob + (size_t)me.x * 16;
    // offsets in bytes of the gathered vector: 8 (integers) or 4 (FP32) an entry
    if (lane < ring_head(n) / 4) reinterpret_cast<int *>(dst)[lane] = lane < n ? off * (sizeof(VT) == 8 ? 8 : 4) : 0;
    VT *vals = reinterpret_cast<VT *>(dst + ring_head(n)) + lane;
    const long long a = M.ptr[t];
    const int w = (int)((M.ptr[t + 1] - a) >> 5);
    for (int k = 0; k < n; ++k) {
        const int o = __shfl_sync(0xffffffffu, off, k);
        VT v;
        ring_zero(v);
        if (row < M.n)
            for (int e = 0; e < w; ++e) {
                const long long i = a + 32LL * e + lane;
                const int oe = M.cols16 ? (int)M.cols16[i] : M.cols32[i] - row;
                if (oe == o && !(oe == 0 && M.vals[i] == 0.0)) v = ring_convert<VT>(M.vals[i], row, o, c, u);
            }
        vals[32 * k] = v;
    }
}

}  // namespace gbcg
