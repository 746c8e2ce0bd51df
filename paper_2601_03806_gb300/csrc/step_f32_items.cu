// step_f32_items.cu -- the grouped-row kernels (k_step_items) of the FP32 step:
// rows of up to 256 nodes, several to a work item.
#include "step_kernel.cuh"

namespace flbm {

cudaError_t launch_items_f32(float *g, const StepArgs<float> &a, int scheme, bool odd, bool stats, int row_grid,
                             cudaStream_t s)
{
    return launch_items<float, float>(g, a, row_plan<float>(a.nx, a.ny, a.nz), scheme, odd, stats, row_grid, s);
}

int items_resident_f32(int scheme, uint32_t nx, uint32_t ny, uint32_t nz)
{
    return items_resident<float, float>(row_plan<float>(nx, ny, nz), scheme);
}

}  // namespace flbm
