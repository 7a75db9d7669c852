// cg_solve_noalloc: the FP64 CG solve for callers that cannot allocate
// device memory.
//
// Some callers of this library may not call cudaMalloc: code embedded in a
// framework whose caching allocator owns the device memory (a cudaMalloc
// beside it can fail once the framework holds the memory, and it
// synchronizes the whole device), real-time loops whose latency budget has no
// room for the device-wide synchronization an allocation implies, and
// plug-ins that run inside a host application with a fixed device-memory
// budget.  cg_create allocates the matrix copy and the solver workspace, so
// those callers cannot use it.  This entry point takes the matrix and the
// vectors from the caller and keeps its workspace (three vectors, the
// per-CTA partial sums, the grid-barrier counter and the status block) in one
// file-scope __device__ array of fixed size, so it allocates nothing, on the
// device or on the host.  It is synchronous: it returns once the result and
// the status are back.
//
// The workspace array is shared by every call in the process and keeps the
// contents of the last call: each call clears what must start at zero (the
// barrier counter and the status block) and writes every vector entry before
// reading it.  Two calls whose work overlaps on the GPU (on different streams,
// or from different host threads) race on that array.
//
// In host code the array's name only stands for it: its device address is
// looked up with cudaGetSymbolAddress, once per device, with that device
// current, on the device's first call.  With lazy module loading (the CUDA
// default) that first call is also what loads this module on the device and
// so creates the array; make it before any stream capture.  cudaDeviceReset
// destroys the array with the context, so the cached address is stale after
// it: a process that resets a device must not call this entry point on it
// again.
//
// It is textbook CG (q = A p, then x and r, then p: three grid barriers per
// iteration), with the fixed-order sums, thread-0 scalars and bounded barriers
// of the SELL-32 solve kernels, and a row-per-thread SpMV straight from the
// caller's CSR arrays instead of the SELL-32 copy that cg_create builds.  The
// product loads nine entries of a row before their FMAs; x += alpha p runs while
// thread 0 waits for the barrier of r.r.  Per iteration, against two entries in
// flight and 512 threads: 50^3 18.2 us (22.6), 60x61x59 25.9 (29.5), 37x41x29 13.7
// (15.4), 20^3 12.6 (14.0).  A third barrier could be saved with q = A r + beta q
// (17.1, 25.1, 13.0 and 11.7 us), but that q collects the rounding of all
// iterations before it: after 116 iterations at 37x41x29 to 60^3 the iterates were 10 to
// 300 times further from exact ones.
#include <cuda_runtime.h>

#include <climits>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "gbcg.h"
#include "rowwalk.h"
#include "sellsolve.cuh"

using namespace gbcg;

namespace {

constexpr int kNoallocMaxCtas = 256;
constexpr size_t kVecBytes = sizeof(double) * (size_t)CG_NOALLOC_MAX_N;
constexpr size_t kPartialBytes = sizeof(double) * 2 * kNoallocMaxCtas * kRedSlots;
constexpr size_t kOffR = 0;
constexpr size_t kOffP = kOffR + kVecBytes;
constexpr size_t kOffQ = kOffP + kVecBytes;
constexpr size_t kOffPartials = kOffQ + kVecBytes;
constexpr size_t kOffBar = kOffPartials + kPartialBytes;
constexpr size_t kOffStatus = kOffBar + 256;
constexpr size_t kScratchBytes = kOffStatus + 256;
constexpr int kNoallocUnroll = 9;    // entries of a row in flight
constexpr int kNoallocUnroll2 = 7;   // of a lane, two lanes to a row (5: 17.8 us at 50^3, 14: 22.6)
constexpr int kNoallocRows2 = 512;   // rows per CTA from which two lanes share a row

}  // namespace

// The workspace (about 6 MiB); every GPU that loads the library holds it
// until the process exits.
static __device__ __align__(256) unsigned char g_cg_noalloc_scratch[kScratchBytes];

namespace {

struct NoallocArgs {
    int32_t n;
    const int32_t *rowptr;
    const int32_t *colidx;
    const double *vals;
    const double *b;
    double *x;
    double tol;
    int32_t maxit;
};

// Row i's range of entries; false if it is out of bounds.
__device__ __forceinline__ bool noalloc_range(const NoallocArgs &A, int i, int64_t nnz, int &k0, int &k1) {
    k0 = __ldg(A.rowptr + i);
    k1 = __ldg(A.rowptr + i + 1);
    return k0 >= 0 && k1 >= k0 && (int64_t)k1 <= nnz;
}

// sum_k vals[k] v[colidx[k]] over the row's entries, kNoallocUnroll of
// them in flight.  CHECK (the first pass over the matrix): a row range or a
// column out of bounds sets bad and its entries are not read; the passes
// after it run only if there was none.  v is written by this kernel between
// grid barriers: coherent loads.
template <bool CHECK>
__device__ __forceinline__ double noalloc_row(const NoallocArgs &A, int i, const double *v, int64_t nnz,
                                              bool &bad) {
    int k0, k1;
    if (!noalloc_range(A, i, nnz, k0, k1)) {
        bad = true;
        return 0.0;
    }
    double s = 0.0;
    for (RowWalk<kNoallocUnroll> e(k0, k1); e.more(); e.next()) {
        double vr[kNoallocUnroll], xr[kNoallocUnroll];
#pragma unroll
        for (int u = 0; u < kNoallocUnroll; ++u) {
            const bool in = e.has(u);
            vr[u] = in ? __ldg(A.vals + e.k + u) : 0.0;
            const int c = in ? __ldg(A.colidx + e.k + u) : i;
            if (CHECK) {
                const bool ok = (unsigned)c < (unsigned)A.n;
                bad |= !ok;
                xr[u] = ok && in ? __ldca(v + c) : 0.0;
            } else {
                xr[u] = in ? __ldca(v + c) : 0.0;
            }
        }
#pragma unroll
        for (int u = 0; u < kNoallocUnroll; ++u)
            if (e.has(u)) s = fma(vr[u], xr[u], s);
    }
    return s;
}

// Row sums of the warp's 32 rows base .. base + 31 (below row_hi), lane l's
// row's in lane l, two lanes to a row and 16 rows at a time; the partial sums
// are brought together at the end (28 FMAs and an add for 32 rows of 27
// entries instead of 27 FMAs).
//
// Why: with a lane per row a load of the caller's CSR arrays touches 32 lines,
// and the L1 data pipe, not the FP64 pipe, sets the pace once an SM has many
// rows (50^3: it is busy 46% of an iteration, nearly all of the product).  At
// 132651 rows an iteration takes 17.3 us with two lanes and 18.5 with one; at
// 48000 (316 per CTA), where latency counts, 14.0 and 12.6.
__device__ __forceinline__ double noalloc_rows2(const NoallocArgs &A, int base, int row_hi, const double *v) {
    const int lane = threadIdx.x & 31;
    double s[2] = {0.0, 0.0};
    auto row_walk = [&](int row) {
        const bool in = row < row_hi;
        return RowWalk<2 * kNoallocUnroll2>(in ? __ldg(A.rowptr + row) : 0, in ? __ldg(A.rowptr + row + 1) : 0, lane & 1);
    };
    RowWalk<2 * kNoallocUnroll2> e[2] = {row_walk(base + (lane >> 1)), row_walk(base + 16 + (lane >> 1))};
    while (__any_sync(0xffffffffu, e[0].more() || e[1].more())) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            double vr[kNoallocUnroll2], xr[kNoallocUnroll2];
#pragma unroll
            for (int u = 0; u < kNoallocUnroll2; ++u) {
                vr[u] = xr[u] = 0.0;
                if (e[h].has(2 * u)) {
                    vr[u] = __ldg(A.vals + e[h].k + 2 * u);
                    xr[u] = __ldca(v + __ldg(A.colidx + e[h].k + 2 * u));
                }
            }
#pragma unroll
            for (int u = 0; u < kNoallocUnroll2; ++u)
                if (e[h].has(2 * u)) s[h] = fma(vr[u], xr[u], s[h]);
            e[h].next();
        }
    }
    const int src = 2 * (lane & 15);
    const double a0 = __shfl_sync(0xffffffffu, s[0], src), b0 = __shfl_sync(0xffffffffu, s[0], src + 1);
    const double a1 = __shfl_sync(0xffffffffu, s[1], src), b1 = __shfl_sync(0xffffffffu, s[1], src + 1);
    return (lane < 16 ? a0 : a1) + (lane < 16 ? b0 : b1);
}

__global__ void __launch_bounds__(kSellSolveThreads, 1) cg_noalloc_kernel(NoallocArgs A, Params P, int64_t nnz) {
    __shared__ double red[3 * kSellSolveThreads];
    __shared__ double quarter[12];
    __shared__ double bcast[8];
    __shared__ int ctl[16];
    Smem S{};
    S.red = red;
    S.bcast = bcast;
    S.ctl = ctl;
    constexpr int kT = kSellSolveThreads;
    const int tid = threadIdx.x;
    const int G = (int)gridDim.x;
    const int row_lo = (int)((int64_t)A.n * blockIdx.x / G);
    const int row_hi = (int)((int64_t)A.n * (blockIdx.x + 1) / G);
    const bool two = A.n > kNoallocRows2 * G;
    unsigned int epoch = 0;
    int set = 0;
    bool bad = false;
    int status = CG_OK, iters = 0;
    double rr = 0.0, bb = 0.0, rho = 0.0, bnorm = 0.0, tol2bb = 0.0;

    // setup: r = b - A x, p = r; r.r, b.b (and any malformed row)
    double v[3] = {0.0, 0.0, 0.0};
    for (int i = row_lo + tid; i < row_hi; i += kT) {
        const double bi = A.b[i];
        const double ri = bi - noalloc_row<true>(A, i, A.x, nnz, bad);
        P.r[i] = ri;
        P.pd[i] = ri;
        v[0] = fma(ri, ri, v[0]);
        v[1] = fma(bi, bi, v[1]);
    }
    v[2] = __syncthreads_or(bad) ? 1.0 : 0.0;
    block_sum_1k<3>(v, red, quarter);
    // every thread of a CTA has the same v[2]: the CTA's sum is 1024 or 0
    publish_partials<3>(P, set, v);
    if (!grid_barrier<false>(P, epoch, S)) return;
    {
        double t[3];
        grid_totals_1k<3>(P, set, t, quarter);
        set ^= 1;
        if (tid == 0) {
            rr = t[0];
            bb = t[1];
            rho = t[0];
            bnorm = sqrt(bb);
            tol2bb = (P.tol * bnorm) * (P.tol * bnorm);
            int go = 0, zero_b = 0;
            if (t[2] != 0.0) status = CG_EINVAL;
            else if (!finite_bits(bb) || !finite_bits(rr)) status = CG_ENAN;
            else if (bnorm == 0.0) { zero_b = 1; rr = 0.0; }
            else if (rr <= tol2bb) status = CG_OK;
            else go = 1;
            ctl[0] = go;
            ctl[2] = zero_b;
        }
        __syncthreads();
        if (ctl[2])
            for (int i = row_lo + tid; i < row_hi; i += kT) A.x[i] = 0.0;
    }
    if (ctl[0]) {
        if (tid == 0) status = CG_ENOCONV;
        for (int k = 1; k <= P.maxit; ++k) {
            // q = A p, p . q
            double v1[1] = {0.0};
            for (int i = row_lo + tid; i - (tid & 31) < row_hi; i += kT) {
                const double qi = two ? noalloc_rows2(A, i - (tid & 31), row_hi, P.pd)
                                      : (i < row_hi ? noalloc_row<false>(A, i, P.pd, nnz, bad) : 0.0);
                if (i >= row_hi) break;
                P.q[i] = qi;
                v1[0] = fma(P.pd[i], qi, v1[0]);
            }
            block_sum_1k<1>(v1, red, quarter);
            publish_partials<1>(P, set, v1);
            if (!grid_barrier<false>(P, epoch, S)) return;
            double sg[1];
            grid_totals_1k<1>(P, set, sg, quarter);
            set ^= 1;
            if (tid == 0) {
                int go = 0;
                if (!finite_bits(sg[0])) status = CG_ENAN;
                else if (!(sg[0] > 0.0)) status = CG_EBREAKDOWN;
                else go = 1;
                bcast[0] = go ? scalar_quotient(rho, sg[0]) : 0.0;
                ctl[0] = go;
            }
            __syncthreads();
            if (!ctl[0]) break;
            const double alpha = bcast[0];
            // r -= alpha q; r.r
            double v2[1] = {0.0};
            for (int i = row_lo + tid; i < row_hi; i += kT) {
                const double ri = fma(-alpha, P.q[i], P.r[i]);
                P.r[i] = ri;
                v2[0] = fma(ri, ri, v2[0]);
            }
            block_sum_1k<1>(v2, red, quarter);
            publish_partials<1>(P, set, v2);
            // x += alpha p, read by nothing before the end, while thread 0 waits
            grid_arrive(P, epoch);
            if (tid == 0) ctl[15] = grid_wait<false>(P, epoch);
            for (int i = row_lo + tid; i < row_hi; i += kT) A.x[i] = fma(alpha, P.pd[i], A.x[i]);
            __syncthreads();
            if (!ctl[15]) return;
            double t2[1];
            grid_totals_1k<1>(P, set, t2, quarter);
            set ^= 1;
            if (tid == 0) {
                iters = k;
                rr = t2[0];
                int go = 0;
                if (!finite_bits(rr)) status = CG_ENAN;
                else if (rr <= tol2bb) status = CG_OK;
                else if (!(rr > 0.0)) status = CG_EBREAKDOWN;
                else if (k < P.maxit) go = 1;
                if (go) {
                    bcast[1] = scalar_quotient(rr, rho);
                    rho = rr;
                }
                ctl[0] = go;
            }
            __syncthreads();
            if (!ctl[0]) break;
            // p = r + beta p (every gather of it is over), published for the next product
            const double beta = bcast[1];
            for (int i = row_lo + tid; i < row_hi; i += kT) P.pd[i] = fma(beta, P.pd[i], P.r[i]);
            if (!grid_barrier<false>(P, epoch, S)) return;
        }
    }
    if (blockIdx.x == 0 && tid == 0) {
        P.st->iters = iters;
        P.st->rr = rr;
        P.st->bb = bb;
        P.st->true_rr = -1.0;
        atomicCAS(&P.st->status, 0, status);
    }
}

// Device address of the workspace, looked up once per device (with that
// device current) and cached; no allocation.
std::mutex g_setup_mutex;
unsigned char *g_scratch_ptr[128] = {};
int g_grid[128] = {};

int noalloc_setup(int dev, unsigned char **scratch, int *grid) {
    if (dev < 0 || dev >= 128) return CG_EINVAL;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (!g_scratch_ptr[dev]) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_cg_noalloc_scratch) != cudaSuccess || !ptr) return CG_ECUDA;
        if (cudaFuncSetAttribute((const void *)cg_noalloc_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxL1) != cudaSuccess)
            return CG_ECUDA;
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cg_noalloc_kernel,
                                                          kSellSolveThreads, 0) != cudaSuccess ||
            per_sm < 1)
            return CG_ECUDA;
        int g = sms < kNoallocMaxCtas ? sms : kNoallocMaxCtas;
        g_grid[dev] = g;
        g_scratch_ptr[dev] = static_cast<unsigned char *>(ptr);
    }
    *scratch = g_scratch_ptr[dev];
    *grid = g_grid[dev];
    return CG_OK;
}

// True when p points into memory the current device can read in a kernel:
// a device allocation of that device, or managed memory.  Host memory
// (pageable or pinned) and other devices' allocations are refused before any
// launch.  cudaPointerGetAttributes allocates nothing.
bool on_device(const void *p, int dev) {
    cudaPointerAttributes a{};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();   // clear the (non-sticky) error recorded for an unknown pointer
        return false;
    }
    if (a.type == cudaMemoryTypeManaged) return true;
    return a.type == cudaMemoryTypeDevice && a.device == dev;
}

int solve_noalloc(const cg_csr *A, const double *b, double *x, double tol, int32_t maxit, void *stream,
                  cg_info *info);

}  // namespace

// info->status is the return code whether or not the solve ran: a call
// rejected before the solve leaves a result with that status and nothing
// else (relres_true and reverted_at -1).
extern "C" int cg_solve_noalloc(const cg_csr *A, const double *b, double *x, double tol, int32_t maxit,
                                void *stream, cg_info *info) {
    constexpr int32_t kUnset = INT32_MIN;
    if (info) info->status = kUnset;
    const int rc = solve_noalloc(A, b, x, tol, maxit, stream, info);
    if (info) {
        if (info->status == kUnset) {
            *info = cg_info{};
            info->relres_true = -1.0;
            info->reverted_at = -1;
        }
        info->status = rc;
    }
    return rc;
}

namespace {

int solve_noalloc(const cg_csr *A, const double *b, double *x, double tol, int32_t maxit, void *stream,
                  cg_info *info) {
    if (!A || A->mem != CG_MEM_DEVICE) return CG_EINVAL;
    if (A->n < 0 || A->n > CG_NOALLOC_MAX_N || A->nnz < 0 || A->nnz > (int64_t)INT32_MAX) return CG_EINVAL;
    if (!(tol >= 0.0) || !std::isfinite(tol)) return CG_EINVAL;
    if (A->n == 0) {
        if (info) *info = cg_info{0, CG_OK, 0.0, -1.0, 0.0, 0, 0, -1, 0};
        return CG_OK;
    }
    if (!A->rowptr || !b || !x || b == x || (A->nnz > 0 && (!A->colidx || !A->vals))) return CG_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CG_ECUDA;
    if (!on_device(A->rowptr, dev) || !on_device(b, dev) || !on_device(x, dev) ||
        (A->nnz > 0 && (!on_device(A->colidx, dev) || !on_device(A->vals, dev))))
        return CG_EINVAL;
    unsigned char *scratch = nullptr;
    int grid = 0;
    int rc = noalloc_setup(dev, &scratch, &grid);
    if (rc != CG_OK) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(stream);

    NoallocArgs args{A->n, A->rowptr, A->colidx, A->vals, b, x, tol, maxit > 0 ? maxit : A->n};
    Params P{};
    P.n = A->n;
    P.r = reinterpret_cast<double *>(scratch + kOffR);
    P.pd = reinterpret_cast<double *>(scratch + kOffP);
    P.q = reinterpret_cast<double *>(scratch + kOffQ);
    P.partials = reinterpret_cast<double *>(scratch + kOffPartials);
    P.bar = reinterpret_cast<unsigned int *>(scratch + kOffBar);
    P.st = reinterpret_cast<DevStatus *>(scratch + kOffStatus);
    P.tol = tol;
    P.maxit = args.maxit;
    P.phantom = 0;
    P.wait_ns = 5000000000ull;
    int64_t nnz = A->nnz;

    // what must start at zero: the barrier counter and the status block
    cudaError_t e = cudaMemsetAsync(scratch + kOffBar, 0, 256 + 256, st);
    if (e == cudaSuccess) {
        void *kargs[] = {&args, &P, &nnz};
        e = cudaLaunchCooperativeKernel((const void *)cg_noalloc_kernel, dim3(grid), dim3(kSellSolveThreads), kargs, 0,
                                        st);
    }
    DevStatus s{};
    if (e == cudaSuccess) e = cudaMemcpyAsync(&s, scratch + kOffStatus, sizeof(DevStatus), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return CG_ECUDA;
    const double bn = std::sqrt(s.bb);
    if (info) {
        *info = cg_info{};
        info->iters = s.iters;
        info->status = s.status;
        info->relres = bn > 0.0 ? std::sqrt(s.rr) / bn : 0.0;
        info->relres_true = -1.0;
        info->kernel_ms = 0.0;
        info->launches = 1;
        info->outer = 0;
        info->reverted_at = -1;
    }
    return s.status;
}

}  // namespace
