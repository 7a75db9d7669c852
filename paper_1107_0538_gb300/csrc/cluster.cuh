// FP64 CG of small systems inside one thread-block cluster (sm_103a).
//
// What bounds a small system on the whole chip: not its work (at 20^3 a row's
// product is 27 entries on 2 slices per SM) but the two grid-wide sums of an
// iteration, each a barrier through L2 (1.4 us) and a read of every CTA's
// partial sums (1.3 us).  A cluster's barrier takes 0.2 us (375 clocks up to
// 256 threads, 605 at 1024) and a load from another SM's shared memory 270
// clocks, so the solve runs on the up to 16 SMs of one cluster instead, with
// everything an iteration touches on chip:
//   * the CTA's slices of the fixed-point matrix (fixed.cuh) in shared memory
//     for the whole solve, with 16-bit offsets into its window of z;
//   * the window, the rows from its smallest to its largest column: whoever
//     owns a row writes its z into every window that holds it (distributed
//     shared memory);
//   * a row's x, r, z, p and q in its thread's registers;
//   * the sums: the quarter sums of every CTA are written into every CTA's
//     shared memory, and warp 0 of each adds them in the same fixed order.
// Warp 0 is the control warp: it adds the totals and takes the decisions, the
// one after barrier B while the others form the next product.
//
// Measured per iteration (plain CG): 729 rows 4.4 us, on the grid 9.4; 4913
// rows 5.5 against 9.4; 9261 rows 7.0 against 9.9.  What is left: two sums of
// two FP64 butterflies each (541 clocks a butterfly), two cluster barriers and
// a quotient (424 clocks), one after the other.
//
// The recurrence, its stop test and its status codes are cg_sell_kernel's.
// Systems whose slices, windows and sums do not fit 16 SMs' shared memory run
// on the whole grid (plan_cluster in plan.h).
#pragma once

#include "plan.h"
#include "sellsolve.cuh"

namespace gbcg {

struct ClusterArgs {
    const int32_t *__restrict__ cut;   // gridDim.x + 1 slice boundaries
    const int2 *__restrict__ win;      // per CTA: first and past-the-last row of its window
    int32_t entries;                   // padded entries a CTA has room for
    int32_t window;                    // rows of its window
};

// All CTAs of a cluster run at the same time, and every CTA takes every
// branch around these barriers alike (the decisions come from the same totals).
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}

// The address of a shared variable of this CTA in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, int2 v) {
    asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(uint32_t addr, unsigned int v) {
    asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Sums of every thread of the cluster: slot s of quarter g of CTA c.
struct ClusterSlots {
    double v[2][kClusterMaxCtas * 4];   // contiguous
    unsigned int mx[kClusterMaxCtas];
};

// Writes the CTA's quarter sums of v (NV values per thread) and its largest mx
// into `slots` of every CTA of the cluster; the caller's cluster barrier
// publishes them.  Quarter g is added by warp g from the values of the warps
// g, g + 4, ... (FP64 adds on one warp per SM sub-partition).
template <int NV>
__device__ __forceinline__ void cluster_sums(const double (&v)[NV], unsigned int mx, double *red, unsigned int *wmax,
                                             ClusterSlots *slots) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nt = (int)blockDim.x, C = (int)gridDim.x;
    const unsigned int m = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) wmax[w] = m;
#pragma unroll
    for (int j = 0; j < NV; ++j) red[j * nt + threadIdx.x] = v[j];
    __syncthreads();
    if (w < 4) {
        const int me = (int)blockIdx.x;   // one cluster: the CTA's rank
#pragma unroll
        for (int j = 0; j < NV; ++j) {
            double a = 0.0, b = 0.0;
            const double *src = red + j * nt;
            int i = 32 * w + lane;
            if (i < nt) a = src[i];
            for (i += 128; i < nt; i += 256) {
                b += src[i];
                if (i + 128 < nt) a += src[i + 128];
            }
            const double t = warp_sum(a + b);
            if (lane < C) cluster_store(cluster_map(smem_u32(&slots->v[j][4 * me + w]), lane), t);
        }
        if (w == 0) {
            const unsigned int x = __reduce_max_sync(0xffffffffu, lane < nt / 32 ? wmax[lane] : 0u);
            if (lane < C) cluster_store(cluster_map(smem_u32(&slots->mx[me]), lane), x);
        }
    }
}

// Warp 0: the totals, the same bits in every CTA.
template <int NV>
__device__ __forceinline__ void cluster_totals(const ClusterSlots *slots, double (&out)[NV], unsigned int &mx) {
    const int lane = threadIdx.x & 31, C = (int)gridDim.x;
#pragma unroll
    for (int j = 0; j < NV; ++j)
        out[j] = warp_sum((lane < 4 * C ? slots->v[j][lane] : 0.0) + (lane + 32 < 4 * C ? slots->v[j][lane + 32] : 0.0));
    mx = __reduce_max_sync(0xffffffffu, lane < C ? slots->mx[lane] : 0u);
}

template <bool PRE>
__global__ void __launch_bounds__(kSellSolveThreads, 1)
    cg_cluster_kernel(Params P, SellMatrix M, FixedMatrix F, ClusterArgs L) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ ClusterSlots slots_a, slots_b;
    __shared__ unsigned int wmax[32];
    __shared__ double bcast[2];
    __shared__ int ctl[8];
    __shared__ int2 wins[kClusterMaxCtas];
    double *const red = reinterpret_cast<double *>(dyn);   // 2 values per thread
    int2 *const vals = reinterpret_cast<int2 *>(red + 2 * blockDim.x);
    int2 *const zwin = vals + L.entries;
    uint16_t *const offs = reinterpret_cast<uint16_t *>(zwin + L.window);

    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, C = (int)gridDim.x, me = (int)blockIdx.x;
    const int t0 = L.cut[me], t1 = L.cut[me + 1];
    const int t = t0 + w - 1;
    const bool has_slice = w >= 1 && t < t1;   // uniform over the warp; never warp 0
    const int row = t * 32 + lane;
    const bool own = has_slice && row < P.n;
    const int ce = own ? F.c[row] : 0;
    if (tid < C) wins[tid] = L.win[tid];
    // a CTA of fewer than four warps leaves its last quarters at zero
    for (int i = tid; i < 2 * 4 * kClusterMaxCtas; i += (int)blockDim.x)
        slots_a.v[0][i] = slots_b.v[0][i] = 0.0;
    const int wlo = L.win[me].x;

    // this CTA's slices into shared memory
    long long a0 = M.ptr[t0];
    int sa = 0, sw = 0;   // the warp's first entry there, the slice's width
    if (has_slice) {
        const long long a = M.ptr[t];
        sa = (int)(a - a0);
        sw = (int)((M.ptr[t + 1] - a) >> 5);
        for (int k = 0; k < sw; ++k) {
            const int i = sa + 32 * k + lane;
            const int col = row + (int)__ldg(M.cols16 + a0 + i);
            vals[i] = __ldg(F.vals + a0 + i);
            offs[i] = (uint16_t)bchk(col - wlo, L.window);
        }
    }
    // the CTAs whose windows may hold rows of this one
    __syncthreads();
    int d_lo = me, d_hi = me;
    for (int d = 0; d < C; ++d)
        if (wins[d].y > t0 * 32 && wins[d].x < t1 * 32) {
            d_lo = min(d_lo, d);
            d_hi = max(d_hi, d);
        }
    const uint32_t zaddr = smem_u32(zwin);
    auto publish = [&](double z, int S) {
        const int2 v = fixed_publish(z, ce, S);
        for (int d = d_lo; d <= d_hi; ++d) {
            const int2 wd = wins[d];
            if (row >= wd.x && row < wd.y) cluster_store(cluster_map(zaddr + 8u * (unsigned)(row - wd.x), d), v);
        }
    };
    auto bound = [&](double v) { return own ? fixed_ub(v, ce) : 0u; };

    int status = CG_OK, iters = 0;
    double rr = 0.0, bb = 0.0, true_rr = -1.0, rho = 0.0, bnorm = 0.0, tol2bb = 0.0;
    double x = own ? P.x[row] : 0.0, r = 0.0, z = 0.0, p = 0.0, q = 0.0;
    const double dinv = PRE && own ? P.dinv[row] : 1.0;
    unsigned int mz = 0;
    int S = 0;

    // ---- setup: r0 = b - A x0, z0 = M^-1 r0, p0 = z0; r.r, r.z, then b.b
    {
        const double ax = has_slice ? sell_slice_sum(M, t, P.x, 0.0) : 0.0;
        double v[2] = {0.0, 0.0}, u[1] = {0.0};
        if (own) {
            const double bi = P.b[row];
            r = bi - ax;
            z = PRE ? dinv * r : r;
            p = z;
            v[0] = r * r;
            v[1] = r * z;
            u[0] = bi * bi;
        }
        cluster_sync();   // every CTA runs: its shared memory may be written from here on
        cluster_sums<2>(v, bound(z), red, wmax, &slots_a);
        __syncthreads();
        cluster_sums<1>(u, 0u, red, wmax, &slots_b);
        cluster_sync();
        if (w == 0) {
            double ta[2], tb[1];
            unsigned int none;
            cluster_totals<2>(&slots_a, ta, mz);
            cluster_totals<1>(&slots_b, tb, none);
            if (tid == 0) {
                rr = ta[0];
                rho = ta[1];
                bb = tb[0];
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
                ctl[2] = fixed_shift(mz, 0u);
            }
        }
        __syncthreads();
        if (ctl[1]) x = 0.0;   // b = 0: the solution is x = 0
    }

    // ---- the CG loop (every CTA takes the same decisions)
    if (ctl[0]) {
        constexpr int NB = PRE ? 2 : 1;
        S = ctl[2];
        if (own) publish(z, S);
        cluster_sync();
        for (int k = 1;; ++k) {
            // az = A z on warps 1..; warp 0 decides on iteration k - 1 meanwhile
            double az = 0.0;
            if (has_slice) {
                FixedAcc acc;
                const int2 *vv = vals + sa + lane;
                const uint16_t *oo = offs + sa + lane;
#pragma unroll 9
                for (int j = 0; j < sw; ++j) fixed_fma(acc, vv[32 * j], zwin[bchk(oo[32 * j], L.window)]);
                az = fixed_value(acc, ce - F.u - S);
            } else if (w == 0 && k > 1) {
                double t2[NB];
                cluster_totals<NB>(&slots_b, t2, mz);
                if (tid == 0) {
                    iters = k - 1;
                    rr = t2[0];
                    const double rho_new = t2[NB - 1];
                    int go = 0;
                    if (!finite_bits(rr)) status = CG_ENAN;
                    else if (rr <= tol2bb) status = CG_OK;
                    else if (!finite_bits(rho_new)) status = CG_ENAN;
                    else if (!(rho_new > 0.0)) status = CG_EBREAKDOWN;
                    else if (k - 1 < P.maxit) go = 1;   // else ENOCONV
                    if (go) {
                        bcast[1] = scalar_quotient(rho_new, rho);
                        rho = rho_new;
                    }
                    ctl[0] = go;
                }
            }
            __syncthreads();
            if (k > 1 && !ctl[0]) break;
            const double beta = k > 1 ? bcast[1] : 0.0;
            // p = z + beta p, q = A z + beta q (= A p), p . q
            double v1[1] = {0.0};
            unsigned int mq = 0;
            if (own) {
                q = fma(beta, q, az);
                p = fma(beta, p, z);
                v1[0] = p * q;
                mq = fixed_ub(q, ce);
                if (PRE) mq = fixed_ub_mul(mq, dinv);
            }
            cluster_sums<1>(v1, mq, red, wmax, &slots_a);
            cluster_sync();
            if (w == 0) {
                double sg[1];
                cluster_totals<1>(&slots_a, sg, mq);
                if (tid == 0) {
                    int go = 0;
                    if (!finite_bits(sg[0])) status = CG_ENAN;
                    else if (!(sg[0] > 0.0)) status = CG_EBREAKDOWN;
                    else go = 1;
                    const double al = go ? scalar_quotient(rho, sg[0]) : 0.0;
                    bcast[0] = al;
                    ctl[0] = go;
                    ctl[2] = fixed_shift(mz, fixed_ub_mul(mq, al));
                }
            }
            __syncthreads();
            if (!ctl[0]) break;
            const double alpha = bcast[0];
            S = ctl[2];
            // r -= alpha q, z = dinv r (published); r.r, r.z; x += alpha p in the
            // barrier's window
            double v2[NB];
#pragma unroll
            for (int j = 0; j < NB; ++j) v2[j] = 0.0;
            if (own) {
                r = fma(-alpha, q, r);
                z = PRE ? dinv * r : r;
                publish(z, S);
                v2[0] = r * r;
                if constexpr (PRE) v2[NB - 1] = r * z;
            }
            cluster_sums<NB>(v2, bound(z), red, wmax, &slots_b);
            cluster_arrive();
            x = fma(alpha, p, x);
            cluster_wait();
        }
    }

    // ---- publish x, then the true residual ||b - A x||
    if (own) P.x[row] = x;
    if (tid == 0) ctl[3] = (P.true_res && status != CG_ENAN && bb != 0.0) ? 1 : 0;
    __syncthreads();
    if (tid == 0 && P.true_res && status != CG_ENAN && bb == 0.0) true_rr = 0.0;
    cluster_sync();   // every x entry is written
    __threadfence();
    if (ctl[3]) {     // the same in every CTA
        const double ax = has_slice ? sell_slice_sum(M, t, P.x, 0.0) : 0.0;
        double v[1] = {0.0};
        if (own) {
            const double d = P.b[row] - ax;
            v[0] = d * d;
        }
        cluster_sums<1>(v, 0u, red, wmax, &slots_a);
        cluster_sync();   // also: no CTA leaves while its shared memory is written
        if (w == 0) {
            double tt[1];
            unsigned int none;
            cluster_totals<1>(&slots_a, tt, none);
            if (tid == 0) true_rr = tt[0];
        }
    }
    if (me == 0 && tid == 0) {
        P.st->iters = iters;
        P.st->rr = rr;
        P.st->bb = bb;
        P.st->true_rr = true_rr;
        atomicCAS(&P.st->status, 0, status);
    }
}

}  // namespace gbcg
