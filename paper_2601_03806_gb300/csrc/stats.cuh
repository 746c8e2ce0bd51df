// stats.cuh -- accumulation of reduced steps into DevStats (row a9).
#pragma once

#include "internal.h"

namespace flbm {

// red: the NSTAT global sums of one step (StatSlot order) over n nodes.
__device__ __forceinline__ void stats_update(DevStats *st, const double *red, long long step, double n)
{
    for (int s = 0; s < NSTAT; ++s) st->last[s] = red[s];
    for (int a = 0; a < 3; ++a) st->acc_u2[a] += red[S_UX2 + a] / n;
    st->acc_m[0] += red[S_DRHO] / n;
    st->acc_m[1] += (red[S_JX] + red[S_JY] + red[S_JZ]) / n;
    st->acc_m[2] += red[S_M3] / n;
    st->acc_m[3] += red[S_M4] / n;
    for (int k = 0; k < 4; ++k) st->acc_m2[k] += red[S_M1SQ + k] / n;
    st->step = step;
    st->nsamp += 1;
}

// The same for `count` <= kStatSlots consecutive reduced steps, in order, by
// the threads of a CTA: totals[i][NSTAT] of time step[i] (loads bypass the
// L1: other SMs wrote them).  The means are formed in parallel (FP64
// divisions one after the other took most of the time), then a thread per
// accumulator adds them in step order; mean: kStatSlots * kStatTerms doubles
// of shared memory.
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
        double v = __ldcg(r + slot);
        if (t == 4) v = (v + __ldcg(r + S_JY)) + __ldcg(r + S_JZ);
        mean[e] = v / n;
    }
    __syncthreads();
    const int t = threadIdx.x;
    if (t < NSTAT) st->last[t] = __ldcg(totals + (count - 1) * NSTAT + t);
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
