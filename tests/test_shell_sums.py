"""The shells' sums of squares of an FP32 spectrum are as good as sums in FP64,
which the interface promises: 256 squares of random FP32 numbers added in a
chain stay within FP64's own bound, 256 x 2^-53 of the sum, in each of 1000
chains (reference: long double), and so do 16 chains of 16 squares merged.  An
infinite amplitude gives an infinite sum, as FP64 addition does.

The kernel's source, compiled for the host."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_03806_gb300", "csrc")

SRC = r'''
#include <cmath>
#include <cstdint>
#include <cstdio>
#define __host__
#define __device__
#define __forceinline__ inline
#include "error_free.cuh"
using namespace flbm;
static uint64_t state = 88172645463325252ull;
static float draw()   // xorshift (Marsaglia 2003): (-1, 1), magnitudes over twenty binades
{
    state ^= state << 13;
    state ^= state >> 7;
    state ^= state << 17;
    const float v = float(int64_t(state >> 39)) * 0x1p-24f - 1.0f;
    return std::ldexp(v, -int(state % 20));
}
int main()
{
    double chain = 0.0, merged = 0.0;
    for (int trial = 0; trial < 1000; ++trial) {
        ShellSum<float> a, all;
        a.zero();
        all.zero();
        long double exact = 0.0L;
        for (int g = 0; g < 16; ++g) {
            ShellSum<float> part;
            part.zero();
            for (int i = 0; i < 16; ++i) {
                const float v = draw();
                a.add_square(v);
                part.add_square(v);
                exact += (long double)v * v;
            }
            all.add(part);
        }
        const double unit = std::ldexp(double(exact), -53);
        chain = std::fmax(chain, double(std::fabs(a.value() - exact)) / unit);
        merged = std::fmax(merged, double(std::fabs(all.value() - exact)) / unit);
    }
    ShellSum<float> big;
    big.zero();
    big.add_square(1.0f);
    big.add_square(1e30f);
    big.add_square(2.0f);
    big.add(ShellSum<float>(big));
    std::printf("%.3f %.3f %d\n", chain, merged, int(std::isinf(big.value())));
    return 0;
}
'''


def test_sums_of_fp32_squares_keep_fp64_accuracy(tmp_path):
    cxx = shutil.which("g++") or pytest.skip("g++ not found")
    (tmp_path / "main.cpp").write_text(SRC)
    exe = tmp_path / "main"
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(tmp_path / "main.cpp"), "-o",
                    str(exe)], check=True)
    chain, merged, inf = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert float(chain) <= 256
    assert float(merged) <= 256
    assert inf == "1"
