// A lane's walk over the entries [k0, k1) of a CSR row, STEP entries further
// in each step, in unsigned arithmetic and never past the row's end by more
// than a step: with row pointers up to 2^31 - 1, "k + u < k1" for the entries
// of a step, or the step after the last one, leaves the range of an int.  (The
// same walk by a signed count of what is left took cg_solve_noalloc from 18.6
// to 20.9 us per iteration at 50^3.)
#pragma once

#ifdef __CUDACC__
#define GBCG_HD __host__ __device__ __forceinline__
#else
#define GBCG_HD inline
#endif

namespace gbcg {

template <int STEP>
struct RowWalk {
    unsigned int k, end;   // the step's first entry, the row's end

    // From entry k0 + first on (0 <= first < STEP, 0 <= k0 <= k1).
    GBCG_HD RowWalk(int k0, int k1, int first = 0) : k((unsigned)k0 + (unsigned)first), end((unsigned)k1) {}
    GBCG_HD bool more() const { return k < end; }
    GBCG_HD bool has(int d) const { return k + (unsigned)d < end; }   // entry k + d is one of the row's
    GBCG_HD void next() { k = k + STEP < end ? k + STEP : end; }
};

}  // namespace gbcg
