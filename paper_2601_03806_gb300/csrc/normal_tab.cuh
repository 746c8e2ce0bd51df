// normal_tab.cuh -- Box-Muller in FP64 from tables.
//
// The FP64 pipe (two operations per clock and SM) bounds the FP64 step, and
// the library's log and sincospi were two thirds of its operations.  A word
// gives only 2^23 uniforms u = v 2^-24, v odd, so the reductions can be done
// on integers and the FP64 work left is short (Tang's table-driven method,
// ACM TOMS 16, 1990, for both functions):
//   -2 ln u: v = f 2^(e - 23) with f in [2^23, 2^24), x = f 2^-23 in [1, 2); the
//     top nine bits of x pick R, an integer near 2^14 / x, and
//     s = -2 (x R 2^-14 - 1) comes out exactly, |s| < 2^-8; then
//     -2 ln u = K(e) + T + s + s^2 / 4 + s^3 / 12 + ... + s^6 / 192 with K, T =
//     -2 ln of the powers of two and of 2^14 / R as (high, low) parts whose high
//     parts add exactly.  x >= sqrt 2 counts as x / 2 with the next exponent,
//     and the interval at x = 2 has R = 2^13 and T = 0, so the result keeps
//     its relative accuracy as u tends to 1.
//   cos, sin of 2 pi u: the quadrant and the nearest of 1025 table points by
//     integer arithmetic, the rest |d| < 2^-10.3 by two-term series and the
//     addition theorem.
// 11 and 12 FP64 operations; over all 2^23 inputs the results are within 0.75
// units in the last place (-2 ln u) and 1.01 x 2^-53 (cos, sin) of the exact
// ones.
#pragma once

#include <cstdint>

namespace flbm {

struct NormalTab {
    double cs[1025][2];      // cos, sin of (pi / 2) j / 1024
    double logt[512][2];     // T, high and low part, by the top bits of x
    double logk[25][2];      // 2 k ln 2, high and low part
    uint32_t r[512];         // R
};

// Fill the table (host, long double).
inline void build_normal_tab(NormalTab &t);   // normal_tab_host.h

constexpr uint32_t kLogUpper = 212;   // first interval of x >= sqrt 2

#ifdef __CUDA_ARCH__
__device__ __forceinline__ double bits_double(uint64_t b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ uint64_t double_bits(double d) { return uint64_t(__double_as_longlong(d)); }
__device__ __forceinline__ uint32_t float_bits(float f) { return __float_as_uint(f); }
__device__ __forceinline__ float bits_float(uint32_t b) { return __uint_as_float(b); }
__device__ __forceinline__ float rsqrt_seed(float f) { return rsqrtf(f); }
__device__ __forceinline__ int log2_floor(uint32_t v) { return 31 - __clz(int(v)); }
__device__ __forceinline__ void load2(const double (&p)[2], double &a, double &b)
{
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    a = v.x;
    b = v.y;
}
#else
inline double bits_double(uint64_t b)
{
    double d;
    __builtin_memcpy(&d, &b, 8);
    return d;
}
inline uint64_t double_bits(double d)
{
    uint64_t b;
    __builtin_memcpy(&b, &d, 8);
    return b;
}
inline uint32_t float_bits(float f)
{
    uint32_t b;
    __builtin_memcpy(&b, &f, 4);
    return b;
}
inline float bits_float(uint32_t b)
{
    float f;
    __builtin_memcpy(&f, &b, 4);
    return f;
}
inline float rsqrt_seed(float f) { return 1.0f / sqrtf(f); }
inline int log2_floor(uint32_t v) { return 31 - __builtin_clz(v); }
inline void load2(const double (&p)[2], double &a, double &b)
{
    a = p[0];
    b = p[1];
}
#endif

// -2 ln((m + 1/2) 2^-23), m < 2^23.
__host__ __device__ __forceinline__ double neg2_log(const NormalTab &t, uint32_t m)
{
    const uint32_t v = 2u * m + 1u;
    const int e = log2_floor(v);
    const uint32_t f = v << (23 - e);
    const uint32_t i = (f >> 14) & 511u;
    const int k = 24 - e - (i >= kLogUpper ? 1 : 0);
    // 2^16 + x R 2^-13 as bits, x R 2^-13 = f R 2^-36
    const double y = bits_double((uint64_t(1023 + 16) << 52) | (uint64_t(f) * t.r[i]));
    const double s = 65538.0 - y;
    double th, tl, kh, kl;
    load2(t.logt[i], th, tl);
    load2(t.logk[k], kh, kl);
    const double q = fma(fma(fma(fma(1.0 / 192.0, s, 1.0 / 80.0), s, 1.0 / 32.0), s, 1.0 / 12.0), s, 0.25);
    const double p = fma(s * s, q, s);
    return (kh + th) + (p + (kl + tl));
}

// sqrt(t) for t in [2^-24, 2^6] by Goldschmidt's iteration with a final
// correction (Markstein, 2004), from the FP32 reciprocal square root: the
// seed is cut out of t's bits and put back into a double's, so nothing runs
// on the FP64 pipe but the six operations of the iteration.  Within 0.51
// units in the last place over all 2^23 radii.
__host__ __device__ __forceinline__ double sqrt_normal(double t)
{
    const uint64_t b = double_bits(t);
    // a float of t's exponent and leading 23 bits
    const float f = bits_float(uint32_t((b >> 29) - (uint64_t(1023 - 127) << 23)));
    const uint32_t y = float_bits(rsqrt_seed(f));
    const uint64_t yb = (uint64_t(y) << 29) + (uint64_t(1023 - 127) << 52);
    const double r = bits_double(yb);
    const double h0 = bits_double(yb - (uint64_t(1) << 52));   // r / 2
    const double g0 = t * r;
    const double e = fma(-g0, h0, 0.5);
    const double g1 = fma(g0, e, g0), h1 = fma(h0, e, h0);
    return fma(fma(-g1, g1, t), h1, g1);
}

// (ca, sa) = -(cos, sin)(2 pi (m + 1/2) 2^-23), m < 2^23.
__host__ __device__ __forceinline__ void neg_cos_sin(const NormalTab &t, uint32_t m, double &ca, double &sa)
{
    const uint32_t v = 2u * m + 1u, quad = v >> 22, rest = v & 0x3fffffu;
    const uint32_t j = (rest + 2048u) >> 12;
    // d in units of 2 pi 2^-24, an integer in [-2048, 2048]
    const double d = bits_double((uint64_t(1075) << 52) | (rest + 2048u - (j << 12))) - 4503599627372544.0;
    double c, s;
    load2(t.cs[j], c, s);
    // u = 2 pi 2^-24: sin(u d) = d (u - u^3 d^2 / 6), cos(u d) - 1 = d^2 (-u^2 / 2 + u^4 d^2 / 24)
    constexpr double u = 6.2831853071795864769 / 16777216.0;
    const double d2 = d * d;
    const double sd = d * fma(d2, -u * u * u / 6.0, u);
    const double cd = d2 * fma(d2, u * u * u * u / 24.0, -u * u / 2.0);
    const double cc = c + fma(c, cd, -(s * sd));
    const double ss = s + fma(s, cd, c * sd);
    // quadrant: (c, s), (-s, c), (-c, -s), (s, -c), and the overall sign
    const bool odd = quad & 1u;
    const double a = odd ? ss : cc, b = odd ? cc : ss;
    ca = (quad == 0u || quad == 3u) ? -a : a;
    if (odd) ca = quad == 1u ? a : -a;
    sa = quad < 2u ? -b : b;
}

}  // namespace flbm
