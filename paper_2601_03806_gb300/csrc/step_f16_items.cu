// step_f16_items.cu -- the grouped-row kernels (k_step_items) of the FP16-storage step:
// rows of up to 256 nodes, several to a work item.
#include <cuda_fp16.h>

#include "step_kernel.cuh"

namespace flbm {

cudaError_t launch_items_f16(void *g, const StepArgs<float> &a, int scheme, bool odd, bool stats, int row_grid,
                             cudaStream_t s)
{
    return launch_items<__half, float>(static_cast<__half *>(g), a, row_plan<__half>(a.nx, a.ny, a.nz), scheme, odd, stats, row_grid, s);
}

int items_resident_f16(int scheme, uint32_t nx, uint32_t ny, uint32_t nz)
{
    return items_resident<__half, float>(row_plan<__half>(nx, ny, nz), scheme);
}

}  // namespace flbm
