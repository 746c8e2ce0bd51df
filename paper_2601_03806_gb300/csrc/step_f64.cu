// step_f64.cu -- FP64 instantiations of the fused step kernels (parity path:
// double deviations, double arithmetic, normals from tables).
#include "step_kernel.cuh"

namespace flbm {

cudaError_t launch_step_f64(double *g, const StepArgs<double> &a, int scheme, bool odd, bool stats,
                            int grid, int row_grid, cudaStream_t s)
{
    return launch_step_t<double, double, uint64_t>(g, a, scheme, odd, stats, grid, row_grid, s);
}

StepShape step_shape_f64(int scheme, uint32_t nx, uint32_t ny, uint32_t nz, uint64_t, bool stats, int nsm)
{
    return step_shape_t<double, double, uint64_t>(scheme, nx, ny, nz, stats, nsm);
}

}  // namespace flbm
