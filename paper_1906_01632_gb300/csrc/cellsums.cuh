// cellsums.cuh -- weighted sums over the corners of a cell (the Q1 weights of its
// quarter faces) in FP64 and in 64-bit fixed point (bits.cuh).
//
// Header-only, usable from device and host code.
#pragma once

#include <math.h>

#include "bits.cuh"

namespace elder {

// Local corner L = lx + 2 ly + 4 lz of the edge of direction D with
// transverse local position (u, v), at end 0 (A) or 1 (B).
__host__ __device__ constexpr int corner_of(int D, int u, int v, int end)
{
    return D == 0 ? (end + 2 * u + 4 * v)
                  : (D == 1 ? (u + 2 * end + 4 * v) : (u + 2 * v + 4 * end));
}

// y[S][T] = sum_{u,v} (u == S ? 3 : 1) (v == T ? 3 : 1) x[u][v]
template <class R>
__host__ __device__ __forceinline__ void kron31(const R (&x)[2][2], R (&y)[2][2])
{
    R t[2][2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const R a = x[u][0] + x[u][1];
        t[u][0] = R(2) * x[u][0] + a;
        t[u][1] = R(2) * x[u][1] + a;
    }
#pragma unroll
    for (int T_ = 0; T_ < 2; ++T_) {
        const R a = t[0][T_] + t[1][T_];
        y[0][T_] = R(2) * t[0][T_] + a;
        y[1][T_] = R(2) * t[1][T_] + a;
    }
}

// Largest biased exponent of N values, and whether sums in its unit stay in the
// normal range (zeros do; subnormals, infinities, NaN and magnitudes below
// 2^-895 do not: their sums are formed in FP64).
template <int N>
__host__ __device__ __forceinline__ int top_exponent(const double (&x)[N], bool& fits)
{
    int top = 0;
#pragma unroll
    for (int L = 0; L < N; ++L) {
        const int e = biased_exponent(x[L]);
        top = e > top ? e : top;
    }
    fits = top >= 128 && top <= 1900;
    if (top == 0) {
        fits = true;
#pragma unroll
        for (int L = 0; L < N; ++L) fits = fits && (bits_of(x[L]) << 1) == 0;
        top = 1023;
    }
    return top;
}

// Sum of N <= 2^(9 - HEAD) values: in fixed point, else in FP64 in order.
template <int HEAD, int N> __host__ __device__ __forceinline__ double fixed_sum(const double (&x)[N])
{
    bool fits;
    const int top = top_exponent(x, fits);
    if (fits) {
        int64_t a = 0;
#pragma unroll
        for (int L = 0; L < N; ++L) a += to_fixed<HEAD>(x[L], top);
        return from_fixed<HEAD>(a, top);
    }
    double a = x[0];
#pragma unroll
    for (int L = 1; L < N; ++L) a += x[L];
    return a;
}

// kron31 in integers
__host__ __device__ __forceinline__ void kron31(const int64_t (&x)[2][2], int64_t (&y)[2][2])
{
    int64_t t[2][2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int64_t a = x[u][0] + x[u][1];
        t[u][0] = (x[u][0] << 1) + a;
        t[u][1] = (x[u][1] << 1) + a;
    }
#pragma unroll
    for (int T_ = 0; T_ < 2; ++T_) {
        const int64_t a = t[0][T_] + t[1][T_];
        y[0][T_] = (t[0][T_] << 1) + a;
        y[1][T_] = (t[1][T_] << 1) + a;
    }
}

// the 16x-weighted sums of the direction-D edge differences of p
template <int D>
__host__ __device__ __forceinline__ void dir_grad(const double (&p8)[8], double (&gp)[2][2])
{
    double dp[2][2];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v)
            dp[u][v] = p8[corner_of(D, u, v, 1)] - p8[corner_of(D, u, v, 0)];
    kron31(dp, gp);
}

// The same from the corners in fixed point (to_fixed<kHeadP>, top exponent top), for
// cells where that is exact (exact_p): each sum is exact and rounded once, so that it
// is never further off than the FP64 form's.  Differences and weights make 2 x 16: 5
// bits above the 58 of a value.
constexpr int kHeadP = 5;
template <int D>
__host__ __device__ __forceinline__ void dir_grad_fixed(const int64_t (&p8)[8], int top,
                                                                double (&gp)[2][2])
{
    int64_t dp[2][2], g[2][2];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v)
            dp[u][v] = p8[corner_of(D, u, v, 1)] - p8[corner_of(D, u, v, 0)];
    kron31(dp, g);
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) gp[u][v] = from_fixed<kHeadP>(g[u][v], top);
}

// Whether the corners of p are exact in fixed point: no nonzero one lies more than
// kHeadP binary orders below the largest (numbers below 2^-1042 count as zeros).  The
// FP64 form subtracts along the edges first, without error for neighbouring values: a corner
// that loses bits to the unit of a much larger one (the topmost layer of cells, where
// p falls to about 0) would make the flux between two small ones less accurate.
// On the words that hold the exponents, with the sign shifted out: 4 integer
// operations per corner (the residual kernels have few issue slots to spare).
__host__ __device__ __forceinline__ bool exact_p(const double (&p8)[8], int& top)
{
    uint32_t most = 0, least = 0xFFFFFFFFu;
#pragma unroll
    for (int L = 0; L < 8; ++L) {
        const uint32_t w = (uint32_t)(bits_of(p8[L]) >> 32) << 1, v = w - 1;  // (0: the largest v)
        most = w > most ? w : most;
        least = v < least ? v : least;
    }
    top = (int)(most >> 21);
    if (most == 0) {
        top = 1023;
        return true;
    }
    return top >= 128 && top <= 1900 && (int)((least + 1) >> 21) >= top - kHeadP;
}

// Z = (W x W x W) x over the cell's corners L = x + 2 y + 4 z: a (3,1) pass
// along each axis, (a, b) -> (2 a + (a + b), 2 b + (a + b))
__host__ __device__ __forceinline__ void cube31(const double (&x)[8], double (&Z)[8])
{
#pragma unroll
    for (int L = 0; L < 8; ++L) Z[L] = x[L];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int L = 0; L < 8; ++L)
            if (!((L >> d) & 1)) {
                const int H = L | (1 << d);
                const double a = Z[L] + Z[H];
                Z[L] = fma(2.0, Z[L], a);
                Z[H] = fma(2.0, Z[H], a);
            }
}

// In fixed point (to_fixed<kHeadC>): Z has 6 bits, the sum of two 7 above the 55 of a
// value.  A value's bits below 2^-2 of the last bit of the cell's largest are cut off:
// a difference of two entries is off by at most 64 such units before its rounding
// (at most 48 times 2^-53 of the largest value's power of two on random cells, 7 to
// 11 in the root mean square, over uniform values, values over three and twelve
// decades, one large corner and a large plane; the FP64 form, whose entries round at
// up to 64 times that scale, 190 to 380 and 20 to 97).
constexpr int kHeadC = 2;
__host__ __device__ __forceinline__ void cube31(const int64_t (&x)[8], int64_t (&Z)[8])
{
#pragma unroll
    for (int L = 0; L < 8; ++L) Z[L] = x[L];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int L = 0; L < 8; ++L)
            if (!((L >> d) & 1)) {
                const int H = L | (1 << d);
                const int64_t a = Z[L] + Z[H];
                Z[L] = (Z[L] << 1) + a;
                Z[H] = (Z[H] << 1) + a;
            }
}

}  // namespace elder
