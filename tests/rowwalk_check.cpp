// CPU check of csrc/rowwalk.h, built with the undefined-behaviour sanitizer: the
// walks of cg_solve_noalloc's products (one lane or two to a row) visit each
// entry of [k0, k1) once, at the end of the int range too.
#include <climits>
#include <cstdio>
#include <vector>

#include "rowwalk.h"

using namespace gbcg;

// One row by `lanes` lanes of `unroll` entries each per step.
template <int UNROLL, int LANES>
static bool visits_once(int k0, int k1) {
    std::vector<int> seen((size_t)(k1 - k0), 0);
    for (int lane = 0; lane < LANES; ++lane) {
        RowWalk<UNROLL * LANES> e(k0, k1, lane);
        for (int extra = 0; e.more() || extra < 400; e.next()) {   // other lanes may step on
            if (!e.more()) ++extra;
            for (int u = 0; u < UNROLL; ++u)
                if (e.has(LANES * u)) {
                    const unsigned k = e.k + LANES * u;
                    if (k < (unsigned)k0 || k >= (unsigned)k1) return false;
                    ++seen[(size_t)(k - (unsigned)k0)];
                }
        }
    }
    for (int n : seen)
        if (n != 1) return false;
    return true;
}

int main() {
    int bad = 0;
    for (int len = 0; len <= 64; ++len)
        for (int k0 : {0, 1, 1000003, INT_MAX - 64 - len, INT_MAX - 15 - len, INT_MAX - 1 - len, INT_MAX - len}) {
            bad += !visits_once<9, 1>(k0, k0 + len);
            bad += !visits_once<7, 2>(k0, k0 + len);
        }
    std::printf("%d\n", bad);
    return bad != 0;
}
