// normal_tab_host.h -- the values of NormalTab (normal_tab.cuh), formed on the
// host in long double and rounded once.
#pragma once

#include <cmath>

#include "normal_tab.cuh"

namespace flbm {

inline void build_normal_tab(NormalTab &t)
{
    // high parts are multiples of 2^-42: two of them add exactly
    auto split = [](long double v, double (&out)[2]) {
        out[0] = double(std::nearbyint(double(std::ldexp(v, 42)))) * 0x1p-42;
        out[1] = double(v - (long double)out[0]);
    };
    const long double ln2 = std::log(2.0L), half_pi = std::acos(0.0L);
    for (int j = 0; j <= 1024; ++j) {
        // the smaller of the angle and its complement
        const bool low = j <= 512;
        const long double a = half_pi * (low ? j : 1024 - j) / 1024;
        t.cs[j][low ? 0 : 1] = double(std::cos(a));
        t.cs[j][low ? 1 : 0] = double(std::sin(a));
    }
    for (uint32_t i = 0; i < 512; ++i) {
        const long double x = 1.0L + (i + 0.5L) / 512.0L;
        t.r[i] = i == 511 ? 8192u : uint32_t(std::lround(double(16384.0L / x)));
        const long double y = std::log(16384.0L / t.r[i]) - (i >= kLogUpper ? ln2 : 0.0L);
        split(i == 511 ? 0.0L : -2.0L * y, t.logt[i]);
    }
    for (int k = 0; k <= 24; ++k) split(2.0L * k * ln2, t.logk[k]);
}

}  // namespace flbm
