// CPU check of the integer arithmetic of csrc/fixed.cuh (host code only): for
// random rows of w entries, the limb sums and their conversion against exact
// 128-bit integers and one correctly rounded conversion.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "fixed.cuh"

using namespace gbcg;

static uint64_t state = 1;
static uint64_t rnd() {   // splitmix64
    uint64_t z = (state += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
static double uniform() { return (double)(int64_t)rnd() * 0x1p-63; }
static uint64_t bits(double v) {
    uint64_t u;
    std::memcpy(&u, &v, 8);
    return u;
}

int main() {
    long long bad = 0;
    // rounding and splitting of single values, both ends of the range included
    for (int i = 0; i < 200000; ++i) {
        const double v = std::ldexp(i % 7 == 0 ? (i % 2 ? 1.0 : -1.0) : uniform(), -(int)(rnd() % 70));
        const int top = i % 2 ? kFixedBitsA : kFixedBitsZ;
        const long long f = fixed_of(bits(v), top);
        const long double want = roundl(ldexpl((long double)v, top));   // 64-bit mantissa: exact product
        if ((long double)f != want) ++bad;
        const int2 s = fixed_split(f, kFixedLoBits);
        if ((long long)s.x * (1ll << kFixedLoBits) + s.y != f) ++bad;
        if (s.y < -(1 << (kFixedLoBits - 1)) || s.y >= (1 << (kFixedLoBits - 1))) ++bad;
        if (std::llabs((long long)s.x) > (1ll << (top - kFixedLoBits))) ++bad;
    }
    // rows: random, and the largest entries the bounds allow (w = 31)
    for (int i = 0; i < 100000; ++i) {
        const int w = 1 + (int)(rnd() % kFixedMaxWidth), mode = i % 4;
        long long hh = 0, hl = 0, lh = 0, ll = 0;
        __int128 sum = 0;
        for (int k = 0; k < w; ++k) {
            // a row's |A| sum to at most 2^63: 8 entries at the top of the range
            long long A = mode == 0 && k < 8 ? (1ll << 60) : (long long)(uniform() * 0x1p58);
            if (mode == 0 && k >= 8) A = (1ll << 29) - 1;
            long long Z = mode <= 1 ? (1ll << 59) : (long long)(uniform() * 0x1p59);
            if (mode == 3) Z >>= rnd() % 60;
            const int2 a = fixed_split(A, kFixedLoBits), z = fixed_split(Z, kFixedLoBits);
            // wrap-around would show as a wrong total
            __int128 t[4] = {(__int128)hh + (__int128)a.x * z.x, (__int128)hl + (__int128)a.x * z.y,
                             (__int128)lh + (__int128)a.y * z.x, (__int128)ll + (__int128)a.y * z.y};
            for (const __int128 &q : t)
                if (q > (__int128)INT64_MAX || q < (__int128)INT64_MIN) ++bad;
            hh = (long long)t[0], hl = (long long)t[1], lh = (long long)t[2], ll = (long long)t[3];
            sum += (__int128)A * Z;
        }
        const int k = (int)(rnd() % 200) - 150;
        const uint64_t got = fixed_to_double_bits(hh, hl, lh, ll, k);
        double g;
        std::memcpy(&g, &got, 8);
        // the sum in 64 exact bits plus a remainder: error of one rounding and
        // of the bits below 2^32 units (three truncations)
        const long double hi = (long double)(long long)(sum >> 62) * 0x1p62L,
                          lo = (long double)(long long)(sum & (((__int128)1 << 62) - 1));
        const long double want = ldexpl(hi + lo, k);
        const long double err = fabsl((long double)g - want);
        const long double bar = fabsl(want) * 0x1.01p-53L + ldexpl(1.0L, 34 + k);
        if (!(err <= bar)) ++bad;
    }
    if (fixed_to_double_bits(0, 0, 0, 0, 5) != 0 || fixed_of(bits(0.0), 59) != 0 || fixed_of(bits(-0.0), 59) != 0) ++bad;
    std::printf("%lld\n", bad);
    return bad != 0;
}
