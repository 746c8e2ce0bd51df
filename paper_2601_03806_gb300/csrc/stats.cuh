// stats.cuh -- totals of reduced steps and their accumulation into DevStats
// (row a9).
#pragma once

#include "internal.h"

namespace flbm {

// The sum over nblocks CTAs of one of the NSTAT sums, p[0], p[NSTAT], ..., by
// a CTA of kStatThreads threads in a fixed order (valid in thread 0): every
// entry point's totals have the same bits.  red: kStatThreads doubles of
// shared memory.
constexpr int kStatThreads = 128;
__device__ __forceinline__ double stat_total(const double *p, int nblocks, double *red)
{
    const int t = threadIdx.x;
    double v = 0.0;
#pragma unroll 4
    for (int b = t; b < nblocks; b += kStatThreads) v += p[size_t(b) * NSTAT];
    red[t] = v;
    __syncthreads();
    for (int w = kStatThreads / 2; w > 0; w >>= 1) {
        if (t < w) red[t] += red[t + w];
        __syncthreads();
    }
    return red[0];
}

// Adds `count` <= kStatSlots consecutive reduced steps to st, in order, by the
// threads of a CTA (32 at least): totals[i][NSTAT], in shared memory, are the
// global sums (StatSlot order) over n nodes of time step[i].  The means are
// formed in parallel (FP64 divisions one after the other took most of the
// time), then a thread per accumulator adds them in step order; mean:
// kStatSlots * kStatTerms doubles of shared memory.
constexpr int kStatTerms = 11;   // acc_u2, acc_m, acc_m2
__device__ __forceinline__ void stats_update(DevStats *st, const double *totals, int count, const long long *step,
                                             double n, double *mean)
{
    for (int e = threadIdx.x; e < count * kStatTerms; e += blockDim.x) {
        const int t = e % kStatTerms;
        const double *r = totals + e / kStatTerms * NSTAT;
        const int slot = t < 3   ? S_UX2 + t
                         : t < 7 ? (t == 3 ? S_DRHO : (t == 4 ? S_JX : (t == 5 ? S_M3 : S_M4)))
                                 : S_M1SQ + t - 7;
        mean[e] = (t == 4 ? (r[slot] + r[S_JY]) + r[S_JZ] : r[slot]) / n;
    }
    __syncthreads();
    const int t = threadIdx.x;
    if (t < NSTAT) st->last[t] = totals[(count - 1) * NSTAT + t];
    if (t < kStatTerms) {
        double *acc = t < 3 ? &st->acc_u2[t] : (t < 7 ? &st->acc_m[t - 3] : &st->acc_m2[t - 7]);
        double a = *acc;
        for (int i = 0; i < count; ++i) a += mean[i * kStatTerms + t];
        *acc = a;
    }
    if (t == 31) {
        st->step = step[count - 1];
        st->nsamp += count;
    }
}

}  // namespace flbm
