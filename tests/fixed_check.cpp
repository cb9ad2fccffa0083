// Host check of the fixed-point sums of csrc/bits.cuh against exact sums in
// 128-bit integers: every result within half a unit in the last place of the
// exact sum plus the truncations of its terms.
#include <cmath>
#include <cstdio>
#include <random>

#include "bits.cuh"

using namespace elder;

template <int HEAD> int check(int terms, std::mt19937_64& r)
{
    int bad = 0;
    for (int it = 0; it < 100000; ++it) {
        const int base = (int)(r() % 1500) - 700;  // exponents 2^-700 .. 2^799
        double x[24];
        int top = 0;
        for (int q = 0; q < terms; ++q) {
            const double f = (double)(r() >> 11) * 0x1p-53 - 0.5;
            x[q] = r() % 9 == 0 ? 0.0 : std::ldexp(f, base + (int)(r() % 70) - 60);
            if (biased_exponent(x[q]) > top) top = biased_exponent(x[q]);
        }
        if (top == 0) continue;
        int64_t a = 0;
        long double exact = 0.0L;  // (80 or 128 bits: truncations dominate)
        for (int q = 0; q < terms; ++q) {
            a += to_fixed<HEAD>(x[q], top);
            exact += (long double)x[q];
        }
        const double got = from_fixed<HEAD>(a, top);
        const long double unit = ldexpl(1.0L, top - 1023 - 52 - HEAD);
        const long double bound =
            terms * unit + fabsl(exact) * 0x1p-53L + terms * fabsl(exact) * 0x1p-60L;
        if (fabsl((long double)got - exact) > bound) ++bad;
    }
    return bad;
}

int main()
{
    std::mt19937_64 r(7);
    int bad = check<2>(1, r) + check<4>(2, r) + check<7>(4, r) + check<6>(8, r);
    // exact round trips, signs, zeros, full mantissas that carry
    const double v[] = {1.0, -1.0, 0.1, 1.9999999999999998, -0x1.fffffffffffffp300, 0x1p-700, 3e5};
    for (double x : v) {
        const int t = biased_exponent(x);
        if (from_fixed<4>(to_fixed<4>(x, t), t) != x) ++bad;
        if (from_fixed<4>(to_fixed<4>(x, t + 4), t + 4) != x) ++bad;
    }
    if (to_fixed<4>(0.0, 1023) != 0 || to_fixed<4>(-0.0, 1023) != 0 || from_fixed<2>(0, 1023) != 0.0)
        ++bad;
    if (to_fixed<2>(1.0, 1023 + 63) != 0 || to_fixed<2>(-1.0, 1023 + 200) != 0) ++bad;
    if (from_fixed<2>(INT64_MAX, 1023 + 54) != 0x1p63) ++bad;
    if (biased_exponent(INFINITY) != 2047 || biased_exponent(NAN) != 2047 ||
        biased_exponent(0x1p-1040) != 0)
        ++bad;
    std::printf("%d\n", bad);
    return bad != 0;
}
