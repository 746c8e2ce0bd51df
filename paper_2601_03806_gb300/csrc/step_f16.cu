// step_f16.cu -- FP16-storage instantiations of the fused step kernels:
// half-precision deviations g_i = f_i - w_i rho0 in HBM (108 B per lattice
// update instead of 216 B), FP32 arithmetic, FP64 reductions.
#include <cuda_fp16.h>

#include "step_kernel.cuh"

namespace flbm {

static bool fits32(uint64_t n) { return n * kQ < (1ull << 32); }

cudaError_t launch_step_f16(void *g, const StepArgs<float> &a, int scheme, bool odd, bool stats,
                            int grid, int row_grid, cudaStream_t s)
{
    __half *h = static_cast<__half *>(g);
    if (row_grid > 0) {
        const RowPlan rp = row_plan<__half>(a.nx, a.ny, a.nz);
        if (rp.grouped) return launch_items_f16(g, a, scheme, odd, stats, row_grid, s);
        if (rows_fixed<512>(rp, a.nx)) return launch_rows_f16_nx512(g, a, scheme, odd, stats, row_grid, s);
    }
    if (fits32(a.ns))
        return launch_step_t<__half, float, uint32_t>(h, a, scheme, odd, stats, grid, row_grid, s);
    return launch_step_t<__half, float, uint64_t>(h, a, scheme, odd, stats, grid, row_grid, s);
}

StepShape step_shape_f16(int scheme, uint32_t nx, uint32_t ny, uint32_t nz, uint64_t ns, bool stats, int nsm)
{
    StepShape s = fits32(ns) ? step_shape_t<__half, float, uint32_t>(scheme, nx, ny, nz, stats, nsm)
                             : step_shape_t<__half, float, uint64_t>(scheme, nx, ny, nz, stats, nsm);
    const RowPlan rp = row_plan<__half>(nx, ny, nz);
    if (rp.grouped) {
        s.rows = items_resident_f16(scheme, nx, ny, nz);
        s.work = rp.work;
        s.item = rp.item.rows * nx;
    } else if (s.rows > 0 && rows_fixed<512>(rp, nx)) {
        s.rows = rows_occupancy_f16_nx512(scheme, stats, ny, nz);
    }
    return s;
}

}  // namespace flbm
