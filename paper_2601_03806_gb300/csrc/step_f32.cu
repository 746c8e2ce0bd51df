// step_f32.cu -- FP32 instantiations of the fused step kernels (throughput
// path: float deviations, float arithmetic, FP64 only in the reductions).
// The direct kernel uses 32-bit node offsets when every population index
// fits (27 N < 2^32, e.g. up to 539^3), 64-bit otherwise.
#include "step_kernel.cuh"

namespace flbm {

static bool fits32(uint64_t n) { return n * kQ < (1ull << 32); }

cudaError_t launch_step_f32(float *g, const StepArgs<float> &a, int scheme, bool odd, bool stats,
                            int grid, int row_grid, cudaStream_t s)
{
    if (row_grid > 0) {
        const RowPlan rp = row_plan<float>(a.nx, a.ny, a.nz);
        if (rp.grouped) return launch_items_f32(g, a, scheme, odd, stats, row_grid, s);
        if (rows_paced<float>(rp)) return launch_rows_f32_paced(g, a, scheme, odd, stats, row_grid, s);
    }
    if (fits32(a.ns))
        return launch_step_t<float, float, uint32_t>(g, a, scheme, odd, stats, grid, row_grid, s);
    return launch_step_t<float, float, uint64_t>(g, a, scheme, odd, stats, grid, row_grid, s);
}

StepShape step_shape_f32(int scheme, uint32_t nx, uint32_t ny, uint32_t nz, uint64_t ns, bool stats, int nsm)
{
    StepShape s = fits32(ns) ? step_shape_t<float, float, uint32_t>(scheme, nx, ny, nz, stats, nsm)
                             : step_shape_t<float, float, uint64_t>(scheme, nx, ny, nz, stats, nsm);
    const RowPlan rp = row_plan<float>(nx, ny, nz);
    if (rp.grouped) {
        s.rows = items_resident_f32(scheme, nx, ny, nz);
        s.work = rp.work;
        s.item = rp.item.rows * nx;
    } else if (rows_paced<float>(rp)) {
        s.rows = rows_occupancy_f32_paced(scheme, stats, nx, ny, nz);
    }
    return s;
}

}  // namespace flbm
