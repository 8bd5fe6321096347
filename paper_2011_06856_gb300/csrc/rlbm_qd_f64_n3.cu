// Quadrant step kernel instances: FP64 storage, N = 3.
#include "rlbm_quad64.cuh"
namespace rlbmk {
cudaError_t launch_quad_f64_n3(int PP, bool one_row, dim3 block, cudaStream_t st, const KernelArgs &a)
{
    return launch_quad64_n<3>(PP, one_row, block, st, a);
}
} // namespace rlbmk
