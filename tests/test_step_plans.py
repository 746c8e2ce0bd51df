"""The launch plans of the step kernels, on the host (the kernels' own header).

* Grouped rows: for every row length they serve and 1 to 40 rows a plane, the
  items of a plane hold 1 to 512 / nx rows each and all of its rows once.
* FP64 boxes of up to 32 nodes per SM share an SM's warps, whatever the number
  of SMs.
* Small boxes: at most 2048 CTAs, the slots that the call without allocation has."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r'''
#include <cstdio>
#include "step_kernel.cuh"
namespace flbm { bool row_pairs_enabled() { return true; } }
using namespace flbm;
template <typename S> void rows()
{
    for (uint32_t nx = 32; nx <= 256; nx += 32)
        for (uint32_t ny = 1; ny <= 40; ++ny) {
            const RowPlan p = row_plan<S>(nx, ny, 3);
            std::printf("rows %u %u %d %u %u %llu\n", nx, ny, int(p.use && p.grouped), p.item.rows, p.item.per_plane,
                        (unsigned long long)p.work);
        }
}
int main()
{
    rows<float>();
    rows<__half>();
    for (uint32_t nsm : {1u, 64u, 132u, 152u, 160u})
        std::printf("few %u %d %d %d\n", nsm, int(direct_plan<double>(32 * nsm, nsm).few),
                    int(direct_plan<double>(32 * nsm + 1, nsm).few), int(direct_plan<float>(1, nsm).few));
    for (uint64_t n : {1ull, 33ull, 65535ull})
        std::printf("ctas %llu %llu\n", (unsigned long long)n, (unsigned long long)direct_plan<float>(n, 152).ctas);
    return 0;
}
'''


def test_plans(tmp_path):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc") or pytest.skip("nvcc not found")
    (tmp_path / "plans.cu").write_text(SRC)
    exe = tmp_path / "plans"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                    "-I" + os.path.join(ROOT, "paper_2601_03806_gb300", "csrc"), str(tmp_path / "plans.cu"), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")
    seen = {"rows": 0, "few": 0, "ctas": 0}
    for line in filter(None, out):
        kind, *v = line.split()
        v = [int(x) for x in v]
        seen[kind] += 1
        if kind == "rows":
            nx, ny, grouped, rows, per_plane, work = v
            assert grouped and 1 <= rows <= min(ny, 512 // nx)
            assert (per_plane - 1) * rows < ny <= per_plane * rows and work == 3 * per_plane
        elif kind == "few":
            assert v[1:] == [1, 0, 0]
        else:
            assert v[1] == -(-v[0] // 32) <= 2048
    assert seen == {"rows": 640, "few": 5, "ctas": 3}
