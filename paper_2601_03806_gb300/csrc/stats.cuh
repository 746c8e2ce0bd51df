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

// The same for `count` consecutive reduced steps, in order: totals[i][NSTAT]
// of time step[i], a thread t per component (at least 32 threads call it;
// the loads bypass the L1, other SMs wrote them).
__device__ __forceinline__ void stats_update(DevStats *st, const double *totals, int count, const long long *step,
                                             double n, int t)
{
    if (t < NSTAT) st->last[t] = __ldcg(totals + (count - 1) * NSTAT + t);
    if (t < 11) {
        // accumulator t and the sums it takes
        double *acc = t < 3 ? &st->acc_u2[t] : (t < 7 ? &st->acc_m[t - 3] : &st->acc_m2[t - 7]);
        const int slot = t < 3   ? S_UX2 + t
                         : t < 7 ? (t == 3 ? S_DRHO : (t == 4 ? S_JX : (t == 5 ? S_M3 : S_M4)))
                                 : S_M1SQ + t - 7;
        double a = *acc;
        for (int i = 0; i < count; ++i) {
            const double *r = totals + i * NSTAT;
            double v = __ldcg(r + slot);
            if (t == 4) v = (v + __ldcg(r + S_JY)) + __ldcg(r + S_JZ);
            a += v / n;
        }
        *acc = a;
    }
    if (t == 31) {
        st->step = step[count - 1];
        st->nsamp += count;
    }
}

}  // namespace flbm
