// Host check of the cell sums of csrc/cellsums.cuh against exact sums in 113-bit
// arithmetic (cells whose values spread over at most 40 binary orders: the sums are
// exact there).
//  p: every weighted difference that the residual uses is as close to the exact one
//     as the FP64 form's, in every cell.
//  c: over each kind of cell, the differences of the cube transform are no further
//     off than the FP64 form's, at most and in the root mean square.
//  porosity: likewise the sums of eight.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>

#include "cellsums.cuh"

using namespace elder;

#if defined(__SIZEOF_FLOAT128__)
typedef __float128 Wide;
#else
typedef long double Wide;  // (113 bits on AArch64)
#endif

static double off(double got, Wide exact)
{
    const Wide d = (Wide)got - exact;
    return (double)(d < 0 ? -d : d);
}

static Wide grad(int D, int S, int T, const double (&p)[8])
{
    Wide a = 0;
    for (int u = 0; u < 2; ++u)
        for (int v = 0; v < 2; ++v)
            a += (Wide)((u == S ? 3 : 1) * (v == T ? 3 : 1)) *
                 ((Wide)p[corner_of(D, u, v, 1)] - (Wide)p[corner_of(D, u, v, 0)]);
    return a;
}

static Wide cube(int L, const double (&c)[8])
{
    Wide a = 0;
    for (int q = 0; q < 8; ++q)
        a += (Wide)((((q ^ L) & 1) ? 1 : 3) * (((q ^ L) & 2) ? 1 : 3) * (((q ^ L) & 4) ? 1 : 3)) *
             (Wide)c[q];
    return a;
}

struct Errors {
    double most = 0.0, square = 0.0;
    void add(double e)
    {
        most = std::max(most, e);
        square += e * e;
    }
};

template <int D> static void check_p(const double (&p)[8], long& worse, long& fixed)
{
    double g64[2][2], g[2][2];
    int64_t P[8];
    int top;
    if (!exact_p(p, top)) return;  // (the FP64 form is taken)
    ++fixed;
    for (int q = 0; q < 8; ++q) P[q] = to_fixed<kHeadP>(p[q], top);
    dir_grad<D>(p, g64);
    dir_grad_fixed<D>(P, top, g);
    for (int S = 0; S < 2; ++S)
        for (int T = 0; T < 2; ++T) {
            const Wide e = grad(D, S, T, p);
            worse += off(g[S][T], e) > off(g64[S][T], e);
        }
}

int main()
{
    std::mt19937_64 r(11);
    std::uniform_real_distribution<double> U(0.0, 1.0);
    int bad = 0;
    for (int kind = 0; kind < 8; ++kind) {
        long worse = 0, fixed = 0;
        Errors c64, c, f64, f;
        const int cells = 10000;
        for (int it = 0; it < cells; ++it) {
            double x[8], p[8];
            const int big = (int)(r() % 8), axis = (int)(r() % 3);
            const double base = U(r);
            for (int q = 0; q < 8; ++q) {
                switch (kind) {
                case 0: x[q] = U(r); break;                                  // uniform
                case 1: x[q] = std::pow(10.0, -12.0 * U(r)); break;          // twelve decades
                case 2: x[q] = std::pow(10.0, -3.0 * U(r)); break;           // three
                case 3: x[q] = q == big ? U(r) : 1e-5 * U(r); break;         // a large corner
                case 4: x[q] = ((q >> axis) & 1) ? U(r) : 1e-3 * U(r); break;  // a large plane
                case 5: x[q] = base * (1.0 + 0.05 * U(r)); break;            // smooth
                case 6: x[q] = r() % 3 ? U(r) : 0.0; break;                  // zeros
                default: x[q] = (r() % 5 ? 1.0 : -0.01) * U(r); break;       // some negative
                }
                // p: hydrostatic and its topmost layer, where it falls to about 0; the
                // last: nearly equal small corners under a large plane
                const double z = (double)(q >> 2);
                p[q] = kind == 0 ? 5e5 + 9.2e4 * (1.0 - z) + 2e3 * x[q]
                     : kind == 1 ? (z > 0 ? 200.0 * (U(r) - 0.5) : 9.2e4 + 2e3 * U(r))
                     : kind == 5 ? (z > 0 ? 100.0 + std::ldexp((double)(r() % 8), -46) : 9.2e4)
                                 : 1e6 * x[q];
            }
            check_p<0>(p, worse, fixed);
            check_p<1>(p, worse, fixed);
            check_p<2>(p, worse, fixed);
            bool fits;
            const int top = top_exponent(x, fits);
            if (!fits) { ++bad; continue; }
            double Z64[8];
            cube31(x, Z64);
            int64_t X[8], Z[8];
            for (int q = 0; q < 8; ++q) X[q] = to_fixed<kHeadC>(x[q], top);
            cube31(X, Z);
            const double scale = std::ldexp(1.0, 1023 + 53 - top);
            for (int d = 0; d < 3; ++d)
                for (int L = 0; L < 8; ++L)
                    if (!((L >> d) & 1)) {
                        const int H = L | (1 << d);
                        const Wide e = cube(H, x) - cube(L, x);
                        c64.add(scale * off(Z64[H] - Z64[L], e));
                        c.add(scale * off(from_fixed<kHeadC>(Z[H] - Z[L], top), e));
                    }
            double phi[8];
            Wide e = 0;
            double a = 0.0;
            for (int q = 0; q < 8; ++q) {
                phi[q] = std::fabs(x[q]);
                e += (Wide)phi[q];
                a += phi[q];
            }
            f64.add(scale * off(a, e));
            f.add(scale * off(fixed_sum<6>(phi), e));
        }
        const bool ok = worse == 0 && c.most <= c64.most && c.square <= c64.square &&
                        f.most <= f64.most && f.square <= f64.square;
        bad += !ok;
        std::printf("kind %d: p worse %ld (fixed in %.2f of the cells); c %.1f %.2f, FP64 %.1f %.2f; "
                    "phi %.2f %.3f, FP64 %.2f %.3f\n",
                    kind, worse, fixed / (3.0 * cells), c.most, std::sqrt(c.square / (12.0 * cells)),
                    c64.most, std::sqrt(c64.square / (12.0 * cells)), f.most,
                    std::sqrt(f.square / cells), f64.most, std::sqrt(f64.square / cells));
    }
    // infinities, NaN and subnormals take the FP64 form, zeros do not
    int top;
    for (double v : {(double)INFINITY, (double)NAN, 0x1p-1040}) {
        const double p[8] = {1, 2, 3, 4, 5, 6, 7, v};
        bad += exact_p(p, top);
    }
    const double some[8] = {0.0, 2, 3, -0.0, 5, 6, 7, 0.0}, none[8] = {};
    bad += !exact_p(some, top) || !exact_p(none, top);
    std::printf("%d\n", bad);
    return bad != 0;
}
