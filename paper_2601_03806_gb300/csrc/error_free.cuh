// error_free.cuh -- sums whose rounding errors are kept: Knuth's TwoSum and the
// shells' sums of squares.  Device code; the same source compiles on the host.
#pragma once

#ifndef __CUDACC__
#include <cmath>
#endif

namespace flbm {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float eft_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float eft_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float eft_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float eft_fms(float a, float b, float c) { return __fmaf_rn(a, b, -c); }
__device__ __forceinline__ double eft_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double eft_sub(double a, double b) { return __dsub_rn(a, b); }
// packed pairs, each lane rounded once; a - b as fma(b, -1, a)
__device__ __forceinline__ float2 eft_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 eft_sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 eft_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 eft_fms(float2 a, float2 b, float2 c)
{
    return __ffma2_rn(a, b, make_float2(-c.x, -c.y));
}
#else
inline float eft_add(float a, float b) { return a + b; }
inline float eft_sub(float a, float b) { return a - b; }
inline float eft_mul(float a, float b) { return a * b; }
inline float eft_fms(float a, float b, float c) { return fmaf(a, b, -c); }
inline double eft_add(double a, double b) { return a + b; }
inline double eft_sub(double a, double b) { return a - b; }
#endif

// s + e = a + b exactly (round to nearest, no underflow or overflow).
template <typename R>
__host__ __device__ __forceinline__ R two_sum(R a, R b, R &e)
{
    const R s = eft_add(a, b);
    const R bb = eft_sub(s, a);
    e = eft_add(eft_sub(a, eft_sub(s, bb)), eft_sub(b, bb));
    return s;
}

// A sum of squares of T.  FP64 squares add in FP64.  FP32 squares add in three
// FP32 numbers: the first takes the rounded terms, the second their rounding
// errors and the squares', the third, plainly rounded, the second's, so a sum
// of K terms S is within 4 K^3 2^-72 S of the exact one before it is rounded
// to FP64 -- inside FP64's own K 2^-53 S up to 360 terms.  FP64 arithmetic
// runs at two operations per clock and SM and bounded the spectra before.
template <typename V>
struct TripleSum {   // V = float, or float2: two sums, a lane each
    V hi, mid, lo;
    __host__ __device__ __forceinline__ void add(V h, V m)
    {
        V e, r, q;
        hi = two_sum(hi, h, e);
        mid = two_sum(mid, e, r);
        mid = two_sum(mid, m, q);
        lo = eft_add(lo, eft_add(r, q));
    }
    __host__ __device__ __forceinline__ void add_square(V v)
    {
        const V p = eft_mul(v, v);
        add(p, eft_fms(v, v, p));
    }
};
template <typename T> struct ShellSum;
template <> struct ShellSum<float> : TripleSum<float> {
    using TripleSum<float>::add;
    __host__ __device__ __forceinline__ void zero() { hi = mid = lo = 0.0f; }
    __host__ __device__ __forceinline__ void add(const ShellSum &o)
    {
        add(o.hi, o.mid);
        lo += o.lo;
    }
    __host__ __device__ __forceinline__ void scale2()
    {
        hi *= 2.0f;
        mid *= 2.0f;
        lo *= 2.0f;
    }
    // an infinite or undefined sum is hi alone (its rounding errors are undefined)
    __host__ __device__ __forceinline__ double value() const
    {
        return hi - hi == 0.0f ? double(hi) + (double(mid) + double(lo)) : double(hi);
    }
};
template <> struct ShellSum<double> {
    double v;
    __host__ __device__ __forceinline__ void zero() { v = 0.0; }
    __host__ __device__ __forceinline__ void add(const ShellSum &o) { v += o.v; }
    __host__ __device__ __forceinline__ void add_square(double x) { v = fma(x, x, v); }
    __host__ __device__ __forceinline__ void scale2() { v *= 2.0; }
    __host__ __device__ __forceinline__ double value() const { return v; }
};

}  // namespace flbm
