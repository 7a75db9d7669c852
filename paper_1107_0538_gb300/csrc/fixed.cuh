// Exact integer SpMV of the FP64 solve kernels (sm_103a).
//
// What bounds the FP64 product: a GB300 SM issues 2 FP64 FMA per clock, so one
// warp-wide DFMA holds an SM sub-partition's FP64 pipe for 64 cycles, while a
// 32 x 32 + 64 bit integer multiply-add (IMAD.WIDE) holds its pipe for 2
// (measured: 1.6 DFMA against 50 IMAD.WIDE lanes per clock per SM in a short
// probe).  Four of them multiply a 60-bit by a 59-bit integer, so the sum of
// a row's products is formed in integers, exactly, at an eighth of the FP64
// pipe's time.
//
// Representation (all powers of two, so scaling is exact):
//   matrix   a_ij = 2^(c_i + c_j - u) A_ij, c_i = about log2(a_ii) / 2, u such
//            that |A_ij| <= 2^60 and a row's |A_ij| sum to at most 2^63;
//            A_ij = a1 2^30 + a0, |a0| <= 2^29
//   vector   Z_j = rint(z_j 2^(c_j + S)), |Z_j| <= 2^59, S the same for the
//            whole vector; Z_j = z1 2^30 + z0, |z0| <= 2^29
//   row      (A z)_i = 2^(c_i - u - S) sum_j A_ij Z_j
// The products with a0 are at most 2^58 each and those with a1 at most 2^29
// times a row sum of 2^33, so a row of up to kFixedMaxWidth = 31 nonzeros stays
// below 2^63 in each of the four 64-bit accumulators: the sum is exact.  The
// scaling by the diagonal's roots makes every entry of an SPD matrix at most
// about 1 in these units, at material interfaces too.
//
// Measured (FP64 CG at 50^3, per iteration): 13.35 us with the FP64 product,
// 11.2 with this one, where the two grid barriers and the latency of the
// loads are left; Jacobi-PCG on 161820 rows, 22.2 to 18.6 us.
//
// Error: entries of 2^-7 and more of the largest (all of a Q1 matrix but the
// weak couplings at material interfaces) are exact in A, smaller ones are
// rounded to 2^-61 of it; Z is rounded to 2^-60 of the bound on its largest
// entry, so an entry more than 2^7 smaller has fewer than FP64's 53 bits; the
// sum is rounded once.  Against iterates and solutions in extended precision
// (144 solves of Q1 boxes of 16^3 to 26^3, contrast 1 to 1e3, plain and Jacobi,
// 100 iterations or to 1e-10) the error is 0.19 times the FP64 product's in the
// geometric mean and smaller in 130 of them.  It is larger in four solves to the
// tolerance at contrast 1e3 (2.3e-12 against 2.2e-11 the most: a solve stops at the
// first residual below it) and in eight where both are below 2e-13.  (An FP64
// reference is itself 5e-13 off at 20^3.)
// With A_ij cut at 57 bits solutions were up to 100 times further: its rounding
// is the same in every iteration.
//
// A matrix with a row of more than 31 nonzeros, a column more than 32767 rows
// away, a diagonal entry that is not positive, a row whose entries sum to more
// than 64 in the scaled units, or a diagonal outside 2^+-200 or spread over
// more than a factor of 2^24 (where the one shift of the whole vector would
// leave the small rows of an unpreconditioned residual few bits) keeps the
// FP64 product (fixed_build.cuh).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "sell.cuh"

namespace gbcg {

constexpr int kFixedMaxWidth = 31;
constexpr int kFixedBitsA = 60, kFixedBitsZ = 59, kFixedLoBits = 30;
constexpr int kFixedMaxC = 100;        // |c_i| at most: every scale below stays a normal FP64 power
constexpr int kFixedSpreadC = 12;      // largest c_i - c_j

struct FixedMatrix {
    const int2 *__restrict__ vals;     // {a1, a0} per padded entry, in the SELL-32 order
    const int16_t *__restrict__ cols;  // the SELL-32 copy's 16-bit column offsets
    const int8_t *__restrict__ c;      // c_i per row
    int32_t u;
};

struct FixedAcc {
    long long hh = 0, hl = 0, lh = 0, ll = 0;   // sums of a1 z1, a1 z0, a0 z1, a0 z0
};

__device__ __forceinline__ void fixed_fma(FixedAcc &s, int2 a, int2 z) {
    s.hh += (long long)a.x * z.x;
    s.hl += (long long)a.x * z.y;
    s.lh += (long long)a.y * z.x;
    s.ll += (long long)a.y * z.y;
}

// v = hi 2^lo_bits + lo with lo in [-2^(lo_bits-1), 2^(lo_bits-1)).
__host__ __device__ __forceinline__ int2 fixed_split(long long v, int lo_bits) {
    const int sh = 32 - lo_bits;
    const int lo = (int)((unsigned)(unsigned long long)v << sh) >> sh;
    return make_int2((int)((v - lo) >> lo_bits), lo);
}

// rint(z 2^sh) (halves away from zero), for |z| 2^sh <= 2^60; integer
// operations only.  Zeros and subnormals give 0.
__host__ __device__ __forceinline__ long long fixed_of(unsigned long long bits, int sh) {
    const int e = (int)(bits >> 52) & 0x7ff;
    if (e == 0) return 0;
    const unsigned long long m = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
    int s = e - 1075 + sh;
    s = s > 9 ? 9 : s;
    unsigned long long v;
    if (s >= 0) v = m << s;
    else v = s < -54 ? 0ull : (m + (1ull << (-s - 1))) >> -s;
    return (long long)(bits >> 63) ? -(long long)v : (long long)v;
}

// The FP64 bits nearest to (hh 2^60 + (hl + lh) 2^30 + ll) 2^k (the bits of
// the sum below 2^32 units are dropped: at least 2^-80 of its largest
// product).  Integer operations only; 0 below the normal range.
__host__ __device__ __forceinline__ unsigned long long fixed_to_double_bits(long long hh, long long hl, long long lh,
                                                                            long long ll, int k) {
    static_assert(kFixedLoBits == 30, "weights below");
    const long long t = (lh >> 2) + (hl >> 2) + (ll >> 32);    // in units of 2^32
    // hh 2^28 + t, 128 bits
    unsigned long long lo = ((unsigned long long)hh << 28) + (unsigned long long)t;
    long long hi = (hh >> 36) + (t >> 63) + (lo < (unsigned long long)t ? 1 : 0);
    const unsigned long long sign = (unsigned long long)hi & 0x8000000000000000ull;
    if (sign) {
        lo = 0ull - lo;
        hi = ~hi + (lo == 0 ? 1 : 0);
    }
    if (hi == 0 && lo == 0) return 0;
    int msb;
    unsigned long long m;   // the leading 64 bits
#ifdef __CUDA_ARCH__
    const int z1 = __clzll(hi), z0 = __clzll((long long)lo);
#else
    const int z1 = hi ? __builtin_clzll((unsigned long long)hi) : 64, z0 = lo ? __builtin_clzll(lo) : 64;
#endif
    if (hi != 0) {   // hi < 2^63: z1 >= 1
        m = ((unsigned long long)hi << z1) | (lo >> (64 - z1));
        msb = 127 - z1;
    } else {
        m = lo << z0;
        msb = 63 - z0;
    }
    const int e = 1023 + msb + 32 + k;
    const unsigned long long mant = (m >> 11) + ((m >> 10) & 1);   // 2^52 <= mant <= 2^53
    if (e < 1) return 0;
    if (e > 2046) return sign | 0x7ff0000000000000ull;
    return sign | (((unsigned long long)(e - 1) << 52) + mant);
}

__device__ __forceinline__ double fixed_value(const FixedAcc &s, int k) {
    return __longlong_as_double((long long)fixed_to_double_bits(s.hh, s.hl, s.lh, s.ll, k));
}

// Entry of the published vector: Z limbs of z at row exponent c and shift S.
__device__ __forceinline__ int2 fixed_publish(double z, int c, int S) {
    return fixed_split(fixed_of((unsigned long long)__double_as_longlong(z), c + S), kFixedLoBits);
}

// Upper bounds of scaled magnitudes, as the upper word of an FP64 number with
// its exponent raised by 128 (ordered like the numbers; 0 for zero and
// subnormals): |v| 2^c is below the number with upper word fixed_ub(v, c).
__device__ __forceinline__ unsigned int fixed_ub(double v, int c) {
    const unsigned int h = (unsigned int)__double2hiint(v) & 0x7fffffffu;
    return h < 0x100000u ? 0u : h + ((unsigned int)(c + 128) << 20) + 1u;
}

// The bound of a product: ub times |f|.
__device__ __forceinline__ unsigned int fixed_ub_mul(unsigned int ub, double f) {
    const unsigned int h = (unsigned int)__double2hiint(f) & 0x7fffffffu;
    if (ub == 0u || h < 0x100000u) return 0u;
    const float m = __uint_as_float(0x3f800000u | ((ub & 0xfffffu) << 3)) *
                    __uint_as_float((0x3f800000u | ((h & 0xfffffu) << 3)) + 8u);    // [1, 4]
    const int e = (int)(ub >> 20) + (int)(h >> 20) - 1023;
    if (e < 1) return 1u;
    return ((unsigned int)min(e, 4000) << 20) + ((__float_as_uint(m) - 0x3f800000u) >> 3) + 2u;
}

// The shift S of a vector whose entries are bounded by a + b.
__device__ __forceinline__ int fixed_shift(unsigned int a, unsigned int b) {
    const unsigned int hi = max(a, b), lo = min(a, b);
    const int d = (int)(hi >> 20) - (int)(lo >> 20);
    const float mh = __uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3));
    const float ml = lo == 0u || d > 60 ? 0.0f : __uint_as_float((0x3f800000u | ((lo & 0xfffffu) << 3)) - ((unsigned)d << 23));
    const float s = (mh + ml) * 1.0000005f;    // [1, 4): one rounding of the sum covered
    const int x = (int)(hi >> 20) - 1023 - 128 + 1 + (int)((__float_as_uint(s) >> 23) - 127u);
    return kFixedBitsZ - max(x, -1200);
}

// Adds M entries from entry k on of lane's row to s, all their loads in flight
// before the products.
// Z is written by this kernel between grid barriers: coherent (L1-cached)
// loads, as in sell_slice_sum_at.
template <int M>
__device__ __forceinline__ void fixed_batch(const int2 *vv, const int16_t *cc, const int2 *zrow, int row, int n,
                                            FixedAcc &s) {
    int2 vr[M], zr[M];
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const int c = __ldcg(cc + j * 32);
        vr[j] = __ldcg(vv + j * 32);
#ifdef GBCG_BOUNDS_CHECK
        zr[j] = __ldca(zrow - row + bchk(row + c, n));
#else
        zr[j] = __ldca(zrow + c);
#endif
    }
#pragma unroll
    for (int j = 0; j < M; ++j) fixed_fma(s, vr[j], zr[j]);
}

// Adds entries k0 <= k < k1 of lane's row in slice t (first entry a) to s, in
// batches of U, then 3, then single entries.
template <int U>
__device__ __forceinline__ void fixed_slice_sum(const FixedMatrix &F, int n, int t, long long a, const int2 *Z,
                                                FixedAcc &s, int k0, int k1) {
    const int lane = threadIdx.x & 31;
    const int row = t * 32 + lane;
    const int2 *vv = F.vals + a + lane + k0 * 32;
    const int16_t *cc = F.cols + a + lane + k0 * 32;
    int m = k1 - k0;
    for (; m >= U; m -= U, vv += U * 32, cc += U * 32) fixed_batch<U>(vv, cc, Z + row, row, n, s);
    if constexpr (U > 3)
        for (; m >= 3; m -= 3, vv += 96, cc += 96) fixed_batch<3>(vv, cc, Z + row, row, n, s);
    for (; m > 0; --m, vv += 32, cc += 32) fixed_batch<1>(vv, cc, Z + row, row, n, s);
}

}  // namespace gbcg
