// Solves whose matrix streams through shared memory slice by slice (sm_103a):
// FP64 CG on the fixed-point matrix (fixed.cuh) of systems larger than a slice
// per warp, and mixed-precision refinement.
//
// What bounds these iterations is the matrix stream, so this layout carries
// fewer bytes than SELL-32 and keeps more of them in flight:
//   * Slices with common offsets.  The rows of a stencil matrix reach the same
//     columns relative to themselves, so a slice of 32 rows stores the union
//     of its rows' offsets once (an int32 per entry column) instead of a
//     16-bit offset per entry; a row without an offset has a zero there.  Per
//     entry 8.1 bytes instead of 10 (fixed point), 4.1 instead of 6 (FP32) or
//     2.1 instead of 4 (BF16).  On Q1 boxes the added zeros are 2% at 100^3.
//     Vectors gathered through it have a margin of zeros on both sides.
//   * A ring of slots.  A slice (offsets, then values, contiguous) is one TMA
//     bulk copy into a slot of shared memory.  The warp that has finished a
//     slice starts the copy of the slice that takes its slot next, also across
//     the end of a pass: the matrix never changes, so the ring fills again
//     while the vector phases and grid barriers run.  A CTA with no more
//     slices than slots copies its matrix once.  A matrix larger than L2
//     streams through it evict-first.
//
// Tried: fetching 20 to 80 MB of the next pass into L2 during the vector phases
// (100^3: 60.5 to 67 us against 60.2 without, when that was the iteration's
// time) and keeping a part of the matrix there with evict-last (30 MB 55.6
// against 57.4, 60 MB 62.8, but 34.8 against 34.7 and 42.1 for FP32
// refinement).  Neither is bound by HBM alone: the instructions of the product
// count as much (the 32-bit gather offsets and the batches without predicates
// took FP32 refinement at 100^3 from 34.7 to 28.6 us).
//
// Warp 0 is the control warp and owns no slice; warp w >= 1 of CTA c owns
// slices w - 1, w - 1 + 31, ... of the CTA's range.  The product needs no beta,
// so after the barrier that publishes z the other warps form their first
// slice's product while warp 0 takes the stop decision.
#pragma once

#include "plan.h"
#include "sellsolve.cuh"

namespace gbcg {

constexpr int kRingWarps = kSellSolveThreads / 32 - 1;   // warps that own slices
constexpr int kRingMaxSlots = 64;
constexpr size_t kRingBytes = 164 * 1024;   // slots of a CTA together; the rest of the 256 KB is L1 for the
                                            // gathered vector (FP64 CG 100^3: 55 us, 128 KB 56, 190 KB 59)
constexpr int kRingRows = 4;     // rows of a thread in flight in the vector phases

struct RingMatrix {
    int32_t n, nslices;
    int32_t slots, slot_bytes;
    int32_t pad;                            // zeros before and after a gathered vector
    int32_t stream;                         // 1: larger than L2, copies marked evict-first
    const int2 *__restrict__ meta;          // per slice: offset in 16-byte units, width
    const unsigned char *__restrict__ blob;
};

__host__ __device__ constexpr int ring_head(int w) { return 16 * ((w + 3) / 4); }   // bytes of the offsets
template <int VB>
__host__ __device__ constexpr int ring_bytes(int w) {
    return w == 0 ? 0 : ring_head(w) + 32 * w * VB;
}

// One CTA's ring.  The copies of a CTA, in the order its slices are used over
// all passes, take the slots in turn; copy g completes phase g / slots of its
// slot's mbarrier.  A slot's slices belong to different warps, and a parity
// wait for a phase is only right once the phase before it is complete; so a
// warp first waits until its copy was started (started[slot] = its phase),
// which the slot's previous user does after its own wait.
template <int VB>
struct Ring {
    const RingMatrix &R;
    unsigned char *smem;
    uint64_t *mbar;
    volatile int *started;   // per slot: phase of the last copy started (shared memory)
    int t0, m;        // first slice of the CTA, their number
    bool resident;    // every slice has a slot of its own: copied once
    int ds, dq;       // slot and phase from one of a warp's slices to its next
    int s0 = 0, q0 = 0;   // slot and phase of the pass's first slice
    int s = 0, q = 0;     // of the warp's current slice

    __device__ __forceinline__ Ring(const RingMatrix &r, unsigned char *s, uint64_t *b, int *l, const int32_t *cut)
        : R(r), smem(s), mbar(b), started(l), t0(cut[blockIdx.x]), m(cut[blockIdx.x + 1] - cut[blockIdx.x]),
          resident(m <= r.slots), ds(kRingWarps % r.slots), dq(kRingWarps / r.slots) {}

    // Starts the copy of slice j into slot s, phase q (one thread).
    __device__ __forceinline__ void issue(int j, int s, int q) const {
        const int2 me = __ldg(R.meta + t0 + j);
        const uint32_t bytes = (uint32_t)ring_bytes<VB>(me.y);
        started[s] = q;
        if (bytes == 0) {
            mbar_arrive(&mbar[s]);
            return;
        }
        mbar_arrive_expect_tx(&mbar[s], bytes);
        const void *src = R.blob + (size_t)me.x * 16;
        tma_load_1d(smem + (size_t)s * R.slot_bytes, src, bytes, &mbar[s], R.stream != 0);
    }

    // Every thread: the barriers, then the first copies.
    __device__ __forceinline__ void start() {
        if (threadIdx.x == 0) {
            for (int i = 0; i < R.slots; ++i) {
                mbar_init(&mbar[i], 1);
                started[i] = -1;
            }
            mbar_init_fence();
        }
        __syncthreads();
        if ((int)threadIdx.x < min(R.slots, m)) issue((int)threadIdx.x, (int)threadIdx.x, 0);
    }

    // The warp's first slice of a pass (j < m), or its next one.
    __device__ __forceinline__ void first(int j) {
        s = resident ? j : s0 + j;
        q = resident ? 0 : q0;
        while (s >= R.slots) s -= R.slots, ++q;
    }
    __device__ __forceinline__ void next() {
        if (resident) {
            s += kRingWarps;
            return;
        }
        s += ds;
        q += dq;
        if (s >= R.slots) s -= R.slots, ++q;
    }

    // The slot of the warp's current slice, once its copy is there; nullptr if
    // the wait ran out (the whole warp).
    __device__ __forceinline__ const unsigned char *wait(unsigned long long limit_ns) const {
        bool ok = true;
        if (started[s] != q) {
            const unsigned long long t = global_ns();
            while (started[s] != q && ok) {
                __nanosleep(64);
                ok = global_ns() - t <= limit_ns;
            }
        }
        ok = ok && mbar_wait_bounded(&mbar[s], (uint32_t)q & 1u, limit_ns);
        return __any_sync(0xffffffffu, !ok) ? nullptr : smem + (size_t)s * R.slot_bytes;
    }

    // The warp is done with slice j, its current one: starts the copy its slot
    // takes next.
    __device__ __forceinline__ void release(int j) const {
        if (resident) return;
        // the lanes' reads of the slot before the async-proxy copy into it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if ((threadIdx.x & 31) == 0) {
            const int n = j + R.slots;   // m > slots: at most one wrap
            issue(n < m ? n : n - m, s, q + 1);
        }
        __syncwarp();
    }

    __device__ __forceinline__ void next_pass() {
        if (resident) return;
        const int g = s0 + m;
        q0 += g / R.slots;
        s0 = g % R.slots;
    }

    // Every thread, before the kernel ends: waits (bounded) for the copies in
    // flight.
    __device__ __forceinline__ void drain(const Params &P) {
        __syncthreads();
        const int i = (int)threadIdx.x;
        if (i < min(R.slots, m) && !mbar_wait_bounded(&mbar[i], (uint32_t)started[i] & 1u, P.wait_ns))
            set_error(P.st, CG_ETIMEOUT, 3);
        __syncthreads();
    }
};

// Index of a gathered vector entry (the vector starts `pad` zeros in).
__device__ __forceinline__ int ring_index(const RingMatrix &R, int i) {
    return bchk(R.pad + i, R.n + 2 * R.pad);
}

// The gathered entry at byte offset `at` of a padded vector: a 32-bit offset
// from a uniform base, so an entry costs one add besides its load.
template <class T>
__device__ __forceinline__ T ring_gather(const RingMatrix &R, const T *z, unsigned int at) {
#ifdef GBCG_BOUNDS_CHECK
    return __ldca(z + bchk((int)(at / sizeof(T)), R.n + 2 * R.pad));
#else
    return __ldca(reinterpret_cast<const T *>(reinterpret_cast<const char *>(z) + at));
#endif
}

__device__ __forceinline__ void ring_fma(FixedAcc &s, int, const int2 *v, int2 z) { fixed_fma(s, *v, z); }
struct LoAcc {
    float s[2] = {0.0f, 0.0f};
};
__device__ __forceinline__ void ring_fma(LoAcc &a, int k, const float *v, float z) { a.s[k & 1] = fmaf(*v, z, a.s[k & 1]); }
__device__ __forceinline__ void ring_fma(LoAcc &a, int k, const __nv_bfloat16 *v, float z) {
    const unsigned int b = *reinterpret_cast<const unsigned short *>(v);
    a.s[k & 1] = fmaf(__uint_as_float(b << 16), z, a.s[k & 1]);
}

// The same for y = A_lo x with a caller's x: a row without the slice's offset
// holds +0 there (and no stored entry is +0, ring_build.cuh), and adds nothing
// even where x is infinite or NaN.  The solve needs no such test: it ends at the
// first sum that is not finite.
struct LoAccStored : LoAcc {};
template <class VT>
__device__ __forceinline__ void ring_fma(LoAccStored &a, int k, const VT *v, float z) {
    bool stored;
    if constexpr (sizeof(VT) == 4) stored = __float_as_uint(*v) != 0u;
    else stored = *reinterpret_cast<const unsigned short *>(v) != 0;
    if (stored) ring_fma(static_cast<LoAcc &>(a), k, v, z);
}

// Whether a slice's value is other than zero.
__device__ __forceinline__ bool ring_adds(int2 v) { return v.x != 0 || v.y != 0; }
__device__ __forceinline__ bool ring_adds(float v) { return v != 0.0f; }
__device__ __forceinline__ bool ring_adds(__nv_bfloat16 v) { return __bfloat162float(v) != 0.0f; }

// Adds the N entries at offs, vals: all gathers in flight, then the products.
template <int N, class VT, class ZT, class Acc>
__device__ __forceinline__ void ring_batch(const RingMatrix &R, const int *offs, const VT *vals, unsigned int rowb,
                                           const ZT *z, Acc &acc) {
    int o[(N + 3) / 4 * 4];
#pragma unroll
    for (int u = 0; u < N; u += 4) *reinterpret_cast<int4 *>(o + u) = *reinterpret_cast<const int4 *>(offs + u);
    ZT zr[N];
#pragma unroll
    for (int u = 0; u < N; ++u) zr[u] = ring_gather(R, z, rowb + (unsigned int)o[u]);
#ifdef GBCG_BOUNDS_CHECK
    for (int u = 0; u < N; ++u)   // an entry that adds something reads a row's value, not the margin
        if (ring_adds(vals[32 * u])) bchk((int)((rowb + (unsigned int)o[u]) / sizeof(ZT)) - R.pad, R.n);
#endif
#pragma unroll
    for (int u = 0; u < N; ++u) ring_fma(acc, u, vals + 32 * u, zr[u]);
}

// Sum of lane's row of the slice in a slot: batches of U entries, then the
// rest of up to U - 1 in two (the branches are the warp's).
template <int U, class VT, class ZT, class Acc>
__device__ __forceinline__ void ring_sum(const RingMatrix &R, const unsigned char *slot, int w, int row, const ZT *z,
                                         Acc &acc) {
    const int *offs = reinterpret_cast<const int *>(slot);
    const VT *vals = reinterpret_cast<const VT *>(slot + ring_head(w)) + (threadIdx.x & 31);
    const unsigned int rowb = (unsigned int)(R.pad + row) * (unsigned int)sizeof(ZT);
    for (; w >= U; w -= U, offs += U, vals += 32 * U) ring_batch<U>(R, offs, vals, rowb, z, acc);
    if (U > 8 && w >= 8) {
        ring_batch<8>(R, offs, vals, rowb, z, acc);
        w -= 8, offs += 8, vals += 256;
    }
    if (w >= 4) {
        ring_batch<4>(R, offs, vals, rowb, z, acc);
        w -= 4, offs += 4, vals += 128;
    }
    if (w == 3) ring_batch<3>(R, offs, vals, rowb, z, acc);
    else if (w == 2) ring_batch<2>(R, offs, vals, rowb, z, acc);
    else if (w == 1) ring_batch<1>(R, offs, vals, rowb, z, acc);
}

// ------------------------------------------------------------- FP64 CG
// The iteration of cg_sellmem_kernel with the fixed-point product; the vectors
// x, r, p and q are in memory (L2), Z (its integers) padded.
template <bool PRE>
__global__ void __launch_bounds__(kSellSolveThreads, 1)
    cg_ring_kernel(Params P, SellMatrix M, RingMatrix R, const int8_t *__restrict__ cexp, int fixed_u, int2 *Z,
                   const int32_t *__restrict__ cut) {
    extern __shared__ __align__(128) unsigned char ring_smem[];
    __shared__ double red[2 * kSellSolveThreads];
    __shared__ double quarter[12];
    __shared__ double bcast[8];
    __shared__ int ctl[16];
    __shared__ unsigned int wmax[kMaxSlots];
    __shared__ uint64_t mbar[kRingMaxSlots];
    __shared__ int started[kRingMaxSlots];
    Smem SM{};
    SM.red = red;
    SM.bcast = bcast;
    SM.ctl = ctl;
    unsigned int epoch = 0;
    int set = 0;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    Ring<8> ring(R, ring_smem, mbar, started, cut);
    ring.start();
    const int t0 = ring.t0, m = ring.m;
    const int j0 = w >= 1 ? w - 1 : m;   // the warp's first slice in the range
    int S = 0;
    unsigned int mz = 0;

    int status = CG_OK, iters = 0;
    double rr = 0.0, bb = 0.0, true_rr = -1.0, rho = 0.0, bnorm = 0.0, tol2bb = 0.0;
    bool timed_out = false;

    // ---- setup: r0 = b - A x0, z0 = M^-1 r0, p0 = z0, q = 0; b.b, then r.r, r.z
    bool run;
    {
        double v[2] = {0.0, 0.0}, vb[1] = {0.0};
        unsigned int mx = 0;
        for (int j = j0; j < m; j += kRingWarps) {
            const int t = t0 + j, row = t * 32 + lane;
            const double ax = sell_slice_sum<kSellUnrollMem>(M, t, P.x, 0.0);
            if (row < P.n) {
                const double bi = P.b[row];
                const double ri = bi - ax;
                const double zi = PRE ? __ldg(P.dinv + row) * ri : ri;
                P.r[row] = ri;
                P.pd[row] = zi;
                P.q[row] = 0.0;
                mx = max(mx, fixed_ub(zi, cexp[row]));
                v[0] = fma(ri, ri, v[0]);
                v[1] = fma(ri, zi, v[1]);
                vb[0] = fma(bi, bi, vb[0]);
            }
        }
        block_sum_1k<1>(vb, red, quarter);
        __syncthreads();
        block_sum_1k<2>(v, red, quarter, wmax, mx);
        const double v3[3] = {v[0], v[1], vb[0]};
        publish_partials<3>(P, set, v3);
        publish_max(P, set, wmax[32]);
        if (!grid_barrier<false>(P, epoch, SM)) goto out;
        double tot[3];
        grid_totals_1k<3>(P, set, tot, quarter, wmax);
        set ^= 1;
        if (tid == 0) {
            rr = tot[0];
            rho = tot[1];
            bb = tot[2];
            bnorm = sqrt(bb);
            tol2bb = (P.tol * bnorm) * (P.tol * bnorm);
            int go = 0, zero_b = 0;
            if (!finite_bits(bb)) {
                status = CG_ENAN;
            } else if (bnorm == 0.0) {
                rr = 0.0;
                zero_b = 1;
            } else if (!finite_bits(rr) || !finite_bits(rho)) {
                status = CG_ENAN;
            } else if (rr <= tol2bb) {
                status = CG_OK;
            } else if (!(rho > 0.0)) {
                status = CG_EBREAKDOWN;
            } else {
                go = 1;
                status = CG_ENOCONV;
            }
            ctl[0] = go;
            ctl[1] = zero_b;
            mz = wmax[33];
            ctl[2] = fixed_shift(mz, 0u);
        }
        __syncthreads();
        run = ctl[0] != 0;
        S = ctl[2];
        for (int j = j0; j < m; j += kRingWarps) {
            const int row = (t0 + j) * 32 + lane;
            if (row >= P.n) continue;
            if (ctl[1]) P.x[row] = 0.0;   // b = 0: the solution is x = 0
            if (run) Z[ring_index(R, row)] = fixed_publish(P.pd[row], cexp[row], S);   // p_0 = z_0
        }
        if (run && !grid_barrier<false>(P, epoch, SM)) goto out;
    }

    // ---- the CG loop
    if (run) {
        constexpr int NB = PRE ? 2 : 1;
        auto decide = [&](int kk, const double (&t2)[NB]) {   // thread 0
            iters = kk;
            rr = t2[0];
            const double rho_new = t2[NB - 1];
            int go = 0;
            if (!finite_bits(rr)) status = CG_ENAN;
            else if (rr <= tol2bb) status = CG_OK;
            else if (!finite_bits(rho_new)) status = CG_ENAN;
            else if (!(rho_new > 0.0)) status = CG_EBREAKDOWN;
            else if (kk < P.maxit) go = 1;   // else ENOCONV
            if (go) {
                bcast[1] = scalar_quotient(rho_new, rho);
                rho = rho_new;
            }
            ctl[0] = go;
        };
        for (int k = 1;; ++k) {
            // phase A: q = A z + beta q (= A p), p = z + beta p; p . q
            double v1[1] = {0.0}, az = 0.0;
            unsigned int mq = 0;
            double qi = 0.0, pi = 0.0, ri = 0.0, di = 1.0;
            int ci = 0;
            auto product = [&](int j) {
                const int t = t0 + j, row = t * 32 + lane;
                const bool in = row < P.n;
                const int2 me = __ldg(R.meta + t);
                if (in) {   // the row's entries, in flight with the wait and the sum
                    qi = P.q[row];
                    pi = P.pd[row];
                    ri = P.r[row];
                    ci = cexp[row];
                    if (PRE) di = __ldg(P.dinv + row);
                }
                const unsigned char *slot = ring.wait(P.wait_ns);
                if (!slot) {
                    timed_out = true;
                    return;
                }
                FixedAcc acc;
                ring_sum<8, int2>(R, slot, me.y, in ? row : P.n - 1, Z, acc);
                ring.release(j);
                az = fixed_value(acc, ci - fixed_u - S);
            };
            if (j0 < m) {
                ring.first(j0);
                product(j0);
            }
            if (w == 0 && k > 1) {
                double t2[NB];
                grid_totals<NB>(P, set ^ 1, t2);
                mz = grid_max(P, set ^ 1);
                if (tid == 0) decide(k - 1, t2);
            }
            if (__syncthreads_or(timed_out)) {
                if (tid == 0) set_error(P.st, CG_ETIMEOUT, 2);
                goto out;
            }
            if (k > 1 && !ctl[0]) break;
            const double beta = k > 1 ? bcast[1] : 0.0;
            for (int j = j0; j < m && !timed_out;) {
                const int row = (t0 + j) * 32 + lane;
                if (row < P.n) {
                    const double zi = PRE ? di * ri : ri;
                    const double qn = fma(beta, qi, az);
                    const double pn = fma(beta, pi, zi);
                    P.q[row] = qn;
                    P.pd[row] = pn;
                    v1[0] = fma(pn, qn, v1[0]);
                    const unsigned int ub = fixed_ub(qn, ci);
                    mq = max(mq, PRE ? fixed_ub_mul(ub, di) : ub);
                }
                j += kRingWarps;
                if (j < m) {
                    ring.next();
                    product(j);
                }
            }
            if (__syncthreads_or(timed_out)) {
                if (tid == 0) set_error(P.st, CG_ETIMEOUT, 2);
                goto out;
            }
            ring.next_pass();
            block_sum_1k<1>(v1, red, quarter, wmax, mq);
            publish_partials<1>(P, set, v1);
            publish_max(P, set, wmax[32]);
            if (!grid_barrier<false>(P, epoch, SM)) goto out;
            double sg[1];
            grid_totals_1k<1>(P, set, sg, quarter, wmax);
            set ^= 1;
            if (tid == 0) {
                const double sigma = sg[0];
                int go = 0;
                if (!finite_bits(sigma)) status = CG_ENAN;
                else if (!(sigma > 0.0)) status = CG_EBREAKDOWN;
                else go = 1;
                const double al = go ? scalar_quotient(rho, sigma) : 0.0;
                bcast[0] = al;
                ctl[0] = go;
                ctl[2] = fixed_shift(mz, fixed_ub_mul(wmax[33], al));
            }
            __syncthreads();
            if (!ctl[0]) break;
            const double alpha = bcast[0];
            S = ctl[2];

            // phase B: r -= alpha q, z = dinv r (its integers published); r.r, r.z
            double v2[NB];
#pragma unroll
            for (int i = 0; i < NB; ++i) v2[i] = 0.0;
            unsigned int mzn = 0;
            for (int j = j0; j < m; j += kRingRows * kRingWarps) {
                // every load of kRingRows rows before the first store
                double qv[kRingRows], rv[kRingRows], dv[kRingRows];
                int cv[kRingRows];
#pragma unroll
                for (int u = 0; u < kRingRows; ++u) {
                    const int ju = j + u * kRingWarps, row = (t0 + ju) * 32 + lane;
                    const bool in = ju < m && row < P.n;
                    qv[u] = in ? P.q[row] : 0.0;
                    rv[u] = in ? P.r[row] : 0.0;
                    cv[u] = in ? cexp[row] : 0;
                    dv[u] = PRE && in ? __ldg(P.dinv + row) : 1.0;
                }
#pragma unroll
                for (int u = 0; u < kRingRows; ++u) {
                    const int ju = j + u * kRingWarps, row = (t0 + ju) * 32 + lane;
                    if (ju < m && row < P.n) {
                        const double rn = fma(-alpha, qv[u], rv[u]);
                        P.r[row] = rn;
                        const double zi = PRE ? dv[u] * rn : rn;
                        Z[ring_index(R, row)] = fixed_publish(zi, cv[u], S);
                        mzn = max(mzn, fixed_ub(zi, cv[u]));
                        v2[0] = fma(rn, rn, v2[0]);
                        if constexpr (PRE) v2[NB - 1] = fma(rn, zi, v2[NB - 1]);
                    }
                }
            }
            block_sum_1k<NB>(v2, red, quarter, wmax, mzn);
            publish_partials<NB>(P, set, v2);
            publish_max(P, set, wmax[32]);
            grid_arrive(P, epoch);
            // x += alpha p, read by nothing before the end, while thread 0 waits
            if (tid == 0) ctl[15] = grid_wait<false>(P, epoch);
            for (int j = j0; j < m; j += kRingRows * kRingWarps) {
                double pv[kRingRows], xv[kRingRows];
#pragma unroll
                for (int u = 0; u < kRingRows; ++u) {
                    const int ju = j + u * kRingWarps, row = (t0 + ju) * 32 + lane;
                    const bool in = ju < m && row < P.n;
                    pv[u] = in ? P.pd[row] : 0.0;
                    xv[u] = in ? P.x[row] : 0.0;
                }
#pragma unroll
                for (int u = 0; u < kRingRows; ++u) {
                    const int ju = j + u * kRingWarps, row = (t0 + ju) * 32 + lane;
                    if (ju < m && row < P.n) P.x[row] = fma(alpha, pv[u], xv[u]);
                }
            }
            __syncthreads();
            if (!ctl[15]) goto out;
            set ^= 1;
        }
    }

    // ---- the true residual ||b - A x||
    {
        if (tid == 0) ctl[3] = (P.true_res && status != CG_ENAN && bb != 0.0) ? 1 : 0;
        __syncthreads();
        if (tid == 0 && P.true_res && status != CG_ENAN && bb == 0.0) true_rr = 0.0;
        if (ctl[3]) {
            if (!grid_barrier<false>(P, epoch, SM)) goto out;   // every x entry is written
            double v[1] = {0.0};
            for (int j = j0; j < m; j += kRingWarps) {
                const int t = t0 + j, row = t * 32 + lane;
                const double ax = sell_slice_sum<kSellUnrollMem>(M, t, P.x, 0.0);
                if (row < P.n) {
                    const double d = P.b[row] - ax;
                    v[0] = fma(d, d, v[0]);
                }
            }
            block_sum_1k<1>(v, red, quarter);
            publish_partials<1>(P, set, v);
            if (!grid_barrier<false>(P, epoch, SM)) goto out;
            double tt[1];
            grid_totals_1k<1>(P, set, tt, quarter);
            if (tid == 0) true_rr = tt[0];
        }
    }

    if (blockIdx.x == 0 && tid == 0) {
        P.st->iters = iters;
        P.st->rr = rr;
        P.st->bb = bb;
        P.st->true_rr = true_rr;
        atomicCAS(&P.st->status, 0, status);
    }
out:
    ring.drain(P);
}

// ------------------------------------------------- mixed precision
// The refinement of cg_irsell_kernel with its inner matrix in the ring: outer
// residual and x in FP64 on the SELL-32 copy, inner CG in FP32 on the
// low-precision slices (diagonal slots -0, the compensated diagonal kept
// apart).  zf: the inner z, padded.
template <class VT>
__global__ void __launch_bounds__(kSellSolveThreads, 1)
    cg_irring_kernel(Params P, SellMatrix M, RingMatrix R, float *zf, const int32_t *__restrict__ cut) {
    extern __shared__ __align__(128) unsigned char ring_smem[];
    __shared__ double red[2 * kSellSolveThreads];
    __shared__ double quarter[12];
    __shared__ double bcast[8];
    __shared__ int ctl[16];
    __shared__ uint64_t mbar[kRingMaxSlots];
    __shared__ int started[kRingMaxSlots];
    Smem SM{};
    SM.red = red;
    SM.bcast = bcast;
    SM.ctl = ctl;
    unsigned int epoch = 0;
    int set = 0;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    Ring<(int)sizeof(VT)> ring(R, ring_smem, mbar, started, cut);
    ring.start();
    const int t0 = ring.t0, m = ring.m;
    const int j0 = w >= 1 ? w - 1 : m;

    int status = CG_ENOCONV, inner_total = 0, outer = 0;   // thread 0's
    double rr = 0.0, bb = 0.0, bnorm = 0.0, rho = 0.0;
    bool timed_out = false;

    for (int o = 0;; ++o) {
        // ---- outer residual in FP64 and the start of the inner solve
        {
            double v[2] = {0.0, 0.0}, vz[1];   // r.r and b.b; r32.z32
            float rz = 0.0f;
            for (int j = j0; j < m; j += kRingWarps) {
                const int t = t0 + j, row = t * 32 + lane;
                const double ax = sell_slice_sum(M, t, P.x, 0.0);
                if (row < P.n) {
                    const double bi = P.b[row];
                    const double ri = bi - ax;
                    v[0] = fma(ri, ri, v[0]);
                    v[1] = fma(bi, bi, v[1]);
                    const float rf = (float)ri;
                    const float z = P.precond ? __ldg(P.dinv32 + row) * rf : rf;
                    P.r32[row] = rf;
                    zf[ring_index(R, row)] = z;
                    P.pd32[row] = z;
                    P.q32[row] = 0.0f;
                    P.d32[row] = 0.0f;
                    rz = fmaf(rf, z, rz);
                }
            }
            vz[0] = (double)rz;
            block_sum_1k<1>(vz, red, quarter);
            __syncthreads();
            block_sum_1k<2>(v, red, quarter);
            const double v3[3] = {v[0], v[1], vz[0]};
            publish_partials<3>(P, set, v3);
            if (!grid_barrier<false>(P, epoch, SM)) goto out;
            double tt[3];
            grid_totals_1k<3>(P, set, tt, quarter);
            set ^= 1;
            if (tid == 0) {
                rr = tt[0];
                if (o == 0) {
                    bb = tt[1];
                    bnorm = sqrt(bb);
                }
                int go = 0, zero_b = 0;
                if (!finite_bits(bb) || !finite_bits(rr) || !finite_bits(tt[2])) status = CG_ENAN;
                else if (bnorm == 0.0) { status = CG_OK; zero_b = 1; rr = 0.0; }
                else if (sqrt(rr) <= P.tol * bnorm) status = CG_OK;
                else if (o == P.max_outer || inner_total >= P.maxit) status = CG_ENOCONV;
                else if (!(tt[2] > 0.0)) status = CG_EBREAKDOWN;
                else go = 1;
                rho = tt[2];                                           // of the inner start
                bcast[2] = (P.inner_tol * P.inner_tol) * tt[0];        // inner target on ||r32||^2
                ctl[0] = go;
                ctl[1] = zero_b;
            }
            __syncthreads();
            if (ctl[1])
                for (int j = j0; j < m; j += kRingWarps)
                    if ((t0 + j) * 32 + lane < P.n) P.x[(t0 + j) * 32 + lane] = 0.0;
            if (!ctl[0]) break;
        }

        // ---- inner CG in FP32 on A_lo d = r (two barriers per iteration)
        for (int k = 1;; ++k) {
            // q = A_lo z + beta q (= A_lo p), p = z + beta p; p . q
            float pq = 0.0f, s = 0.0f, qi = 0.0f, pi = 0.0f, zi = 0.0f, dg = 0.0f;
            auto product = [&](int j) {
                const int t = t0 + j, row = t * 32 + lane;
                const bool in = row < P.n;
                const int2 me = __ldg(R.meta + t);
                if (in) {   // the row's entries, in flight with the wait and the sum
                    qi = P.q32[row];
                    pi = P.pd32[row];
                    zi = zf[ring_index(R, row)];
                    dg = __ldg(P.diag_lo + row);
                }
                const unsigned char *slot = ring.wait(P.wait_ns);
                if (!slot) {
                    timed_out = true;
                    return;
                }
                LoAcc acc;
                ring_sum<16, VT>(R, slot, me.y, in ? row : P.n - 1, zf, acc);
                s = acc.s[0] + acc.s[1];
                ring.release(j);
            };
            if (j0 < m) {
                ring.first(j0);
                product(j0);
            }
            if (w == 0 && k > 1) {
                double t2[2];
                grid_totals<2>(P, set ^ 1, t2);
                if (tid == 0) {   // decision on inner iteration k - 1
                    ++inner_total;
                    int go = 0;
                    if (!finite_bits(t2[0]) || !finite_bits(t2[1]) || !(t2[1] > 0.0)) go = 0;
                    else if (t2[0] <= bcast[2]) go = 0;                 // inner target met
                    else if (k - 1 >= P.max_inner || inner_total >= P.maxit) go = 0;
                    else go = 1;
                    if (go) {
                        bcast[1] = scalar_quotient(t2[1], rho);
                        rho = t2[1];
                    }
                    ctl[0] = go;
                }
            }
            if (__syncthreads_or(timed_out)) {
                if (tid == 0) set_error(P.st, CG_ETIMEOUT, 2);
                goto out;
            }
            const bool stop = k > 1 && !ctl[0];
            const float beta = k > 1 ? (float)bcast[1] : 0.0f;
            // a stopped inner solve still walks the ring to the end of the pass
            for (int j = j0; j < m && !timed_out;) {
                const int row = (t0 + j) * 32 + lane;
                if (!stop && row < P.n) {
                    const float qn = fmaf(beta, qi, fmaf(dg, zi, s));
                    const float pn = fmaf(beta, pi, zi);
                    P.q32[row] = qn;
                    P.pd32[row] = pn;
                    pq = fmaf(pn, qn, pq);
                }
                j += kRingWarps;
                if (j < m) {
                    ring.next();
                    product(j);
                }
            }
            if (__syncthreads_or(timed_out)) {
                if (tid == 0) set_error(P.st, CG_ETIMEOUT, 2);
                goto out;
            }
            ring.next_pass();
            if (stop) break;
            double v1[1] = {(double)pq};
            block_sum_1k<1>(v1, red, quarter);
            publish_partials<1>(P, set, v1);
            if (!grid_barrier<false>(P, epoch, SM)) goto out;
            double sg[1];
            grid_totals_1k<1>(P, set, sg, quarter);
            set ^= 1;
            if (tid == 0) {
                int go = 1;
                if (!finite_bits(sg[0]) || !(sg[0] > 0.0)) go = 0;   // inner breakdown: keep d
                bcast[0] = go ? scalar_quotient(rho, sg[0]) : 0.0;
                ctl[0] = go;
                if (!go && k == 1) status = finite_bits(sg[0]) ? CG_EBREAKDOWN : CG_ENAN;
            }
            __syncthreads();
            if (!ctl[0]) break;
            const float alpha = (float)bcast[0];
            // r -= alpha q, z = M r (published); r.r, r.z; then d += alpha p in the
            // barrier's window
            float prr = 0.0f, prz = 0.0f;
            for (int j = j0; j < m; j += kRingRows * kRingWarps) {
                float qv[kRingRows], rv[kRingRows], dv[kRingRows];
#pragma unroll
                for (int u = 0; u < kRingRows; ++u) {
                    const int ju = j + u * kRingWarps, row = (t0 + ju) * 32 + lane;
                    const bool in = ju < m && row < P.n;
                    qv[u] = in ? P.q32[row] : 0.0f;
                    rv[u] = in ? P.r32[row] : 0.0f;
                    dv[u] = in && P.precond ? __ldg(P.dinv32 + row) : 1.0f;
                }
#pragma unroll
                for (int u = 0; u < kRingRows; ++u) {
                    const int ju = j + u * kRingWarps, row = (t0 + ju) * 32 + lane;
                    if (ju < m && row < P.n) {
                        const float ri = fmaf(-alpha, qv[u], rv[u]);
                        P.r32[row] = ri;
                        prr = fmaf(ri, ri, prr);
                        float z = ri;
                        if (P.precond) {
                            z = dv[u] * ri;
                            prz = fmaf(ri, z, prz);
                        }
                        zf[ring_index(R, row)] = z;
                    }
                }
            }
            double v2[2] = {(double)prr, (double)(P.precond ? prz : prr)};
            block_sum_1k<2>(v2, red, quarter);
            publish_partials<2>(P, set, v2);
            grid_arrive(P, epoch);
            if (tid == 0) ctl[15] = grid_wait<false>(P, epoch);
            for (int j = j0; j < m; j += kRingRows * kRingWarps) {
                float pv[kRingRows], dv[kRingRows];
#pragma unroll
                for (int u = 0; u < kRingRows; ++u) {
                    const int ju = j + u * kRingWarps, row = (t0 + ju) * 32 + lane;
                    const bool in = ju < m && row < P.n;
                    pv[u] = in ? P.pd32[row] : 0.0f;
                    dv[u] = in ? P.d32[row] : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < kRingRows; ++u) {
                    const int ju = j + u * kRingWarps, row = (t0 + ju) * 32 + lane;
                    if (ju < m && row < P.n) P.d32[row] = fmaf(alpha, pv[u], dv[u]);
                }
            }
            __syncthreads();
            if (!ctl[15]) goto out;
            set ^= 1;
        }
        // ---- x += d in FP64
        for (int j = j0; j < m; j += kRingWarps) {
            const int row = (t0 + j) * 32 + lane;
            if (row < P.n) P.x[row] += (double)P.d32[row];
        }
        if (tid == 0) outer = o + 1;
        if (!grid_barrier<false>(P, epoch, SM)) goto out;
    }

    if (blockIdx.x == 0 && tid == 0) {
        P.st->iters = inner_total;
        P.st->outer = outer;
        P.st->rr = rr;
        P.st->bb = bb;
        P.st->true_rr = rr;   // the outer residual is the true FP64 residual
        atomicCAS(&P.st->status, 0, status);
    }
out:
    ring.drain(P);
}

// y = A_lo x alone, through the product of cg_irring_kernel.
template <class VT>
__global__ void __launch_bounds__(kSellSolveThreads, 1)
    lo_spmv_ring_kernel(Params P, RingMatrix R, const float *zf, const int32_t *__restrict__ cut, float *y) {
    extern __shared__ __align__(128) unsigned char ring_smem[];
    __shared__ uint64_t mbar[kRingMaxSlots];
    __shared__ int started[kRingMaxSlots];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Ring<(int)sizeof(VT)> ring(R, ring_smem, mbar, started, cut);
    ring.start();
    const int j0 = w >= 1 ? w - 1 : ring.m;
    if (j0 < ring.m) ring.first(j0);
    for (int j = j0; j < ring.m; j += kRingWarps, ring.next()) {
        const int t = ring.t0 + j, row = t * 32 + lane;
        const unsigned char *slot = ring.wait(P.wait_ns);
        if (!slot) {
            if (lane == 0) set_error(P.st, CG_ETIMEOUT, 2);
            break;
        }
        LoAccStored acc;
        ring_sum<16, VT>(R, slot, __ldg(R.meta + t).y, row < P.n ? row : P.n - 1, zf, acc);
        const float s = acc.s[0] + acc.s[1];
        ring.release(j);
        if (row < P.n) y[row] = fmaf(__ldg(P.diag_lo + row), zf[ring_index(R, row)], s);
    }
    ring.drain(P);
}

}  // namespace gbcg
