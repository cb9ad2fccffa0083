// bits.cuh -- conversions between FP64 and FP32 and magnitude comparisons
// done on the IEEE 754 bit patterns with integer operations.  On GB300 the
// FP64<->FP32 conversion instructions and FP64 min/max issue on the FP64
// pipe, 1/64 of the FP32 rate, which the FP64-bound kernels cannot spare.
//
// Header-only, usable from device and host code (host: plain C++, so that
// the functions are checked on the CPU against the host's own conversions).
#pragma once

#include <stdint.h>
#include <string.h>

#if !defined(__CUDACC__)
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace elder {

__host__ __device__ __forceinline__ uint32_t bits_of(float x)
{
#if defined(__CUDA_ARCH__)
    return __float_as_uint(x);
#else
    uint32_t u;
    memcpy(&u, &x, 4);
    return u;
#endif
}

__host__ __device__ __forceinline__ float float_of(uint32_t u)
{
#if defined(__CUDA_ARCH__)
    return __uint_as_float(u);
#else
    float x;
    memcpy(&x, &u, 4);
    return x;
#endif
}

__host__ __device__ __forceinline__ uint64_t bits_of(double x)
{
#if defined(__CUDA_ARCH__)
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t u;
    memcpy(&u, &x, 8);
    return u;
#endif
}

__host__ __device__ __forceinline__ double double_of(uint64_t u)
{
#if defined(__CUDA_ARCH__)
    return __longlong_as_double((long long)u);
#else
    double x;
    memcpy(&x, &u, 8);
    return x;
#endif
}

// FP32 value of an FP64 number: the exponent rebiased by 127 - 1023, the top
// 23 of the 52 mantissa bits kept (truncated toward zero, not rounded);
// magnitudes below 2^-126 become a zero of the same sign, those from 2^128 up
// (and NaN) infinity.  For the residual's round-off scale, a magnitude needed
// to a few digits, and for powers of two, which it converts exactly.
__host__ __device__ __forceinline__ float d2f_trunc(double x)
{
    const uint64_t u = bits_of(x);
    const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
    const int e = (int)((hi >> 20) & 0x7FFu);
    const uint32_t sign = hi & 0x80000000u;
    uint32_t bits = sign | ((uint32_t)(e - 896) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29);
    bits = e <= 896 ? sign : (e >= 1151 ? (sign | 0x7F800000u) : bits);
    return float_of(bits);
}

// FP64 value of an FP32 number, exact like the conversion instruction:
// exponent rebiased by 1023 - 127, mantissa shifted up by 29 bits; signed
// zeros in the integer path, subnormals, infinities and NaN by the
// conversion itself.
__host__ __device__ __forceinline__ double f2d_exact(float x)
{
    const uint32_t u = bits_of(x), a = u & 0x7FFFFFFFu;
    const uint64_t sign = (uint64_t)(u >> 31) << 63;
    if (a == 0u) return double_of(sign);
    if (a < 0x00800000u || a >= 0x7F800000u) return (double)x;
    return double_of(sign | (((uint64_t)a + (896ull << 23)) << 29));
}

// |x| as its bit pattern, which orders like the magnitude; NaN maps to the
// pattern of +inf
__host__ __device__ __forceinline__ uint32_t mag_bits(float x)
{
    const uint32_t a = bits_of(x) & 0x7FFFFFFFu;
    return a > 0x7F800000u ? 0x7F800000u : a;
}

// ---------------------------------------------------------------------------
// Sums of a few FP64 numbers of one cell in 64-bit integers: the numbers are
// brought to a common power-of-two unit set by the largest exponent among them,
// added and weighted exactly, and each result is rounded once.  A number is cut off
// below 2^-HEAD of the last bit of the largest: numbers within HEAD binary orders of
// it are exact, a smaller one is off by less than that unit, however small it is
// (where FP64 subtracts two small neighbours without error; see cell_p).  FP64
// rounds every operation by up to half the last bit of its own result.
// Integer operations issue at 64 times the FP64 rate here.
// ---------------------------------------------------------------------------

// Biased exponent of x (0 for zeros and subnormals, 2047 for infinities, NaN).
__host__ __device__ __forceinline__ int biased_exponent(double x)
{
    return (int)((uint32_t)(bits_of(x) >> 52) & 0x7FFu);
}

// x in units of 2^(top - 1023 - 52 - HEAD) for biased_exponent(x) <= top < 2047,
// truncated toward zero (exact where the exponents differ by at most HEAD);
// subnormals become 0.  Magnitudes stay below 2^(53 + HEAD).
template <int HEAD> __host__ __device__ __forceinline__ int64_t to_fixed(double x, int top)
{
    const uint64_t u = bits_of(x);
    const int e = (int)((uint32_t)(u >> 52) & 0x7FFu);
    const int s = top - e < 63 ? top - e : 63;
    uint64_t m = ((u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << HEAD;
    m = e == 0 ? 0 : m >> s;
    const int64_t sign = (int64_t)u >> 63;
    return ((int64_t)m ^ sign) - sign;
}

__host__ __device__ __forceinline__ int leading_zeros(uint64_t m)
{
#if defined(__CUDA_ARCH__)
    return __clzll((long long)m);
#else
    return __builtin_clzll(m);
#endif
}

// v units of to_fixed<HEAD>(., top) as FP64, rounded to nearest (halves away
// from zero); |v| < 2^63, and 64 <= top <= 1900, so that no result leaves the
// normal range.
template <int HEAD> __host__ __device__ __forceinline__ double from_fixed(int64_t v, int top)
{
    const uint64_t sign = (uint64_t)v & 0x8000000000000000ull;
    uint64_t m = v < 0 ? (uint64_t)0 - (uint64_t)v : (uint64_t)v;
    const int z = leading_zeros(m | 1);
    m <<= z;  // the leading bit at 63, weight 2^(63 - z) units
    // 53 bits, rounded; the carry of a full mantissa runs into the exponent
    const uint64_t r = (m >> 11) + ((m >> 10) & 1);
    const uint64_t e = (uint64_t)(top - 52 - HEAD + 63 - z - 1);
    return v == 0 ? 0.0 : double_of(sign | ((e << 52) + r));
}

}  // namespace elder
