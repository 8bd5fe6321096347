// Many-angle quadrant step kernel instances: FP32 storage, N = 3.
#include "rlbm_quad_split.cuh"
namespace rlbmk {
cudaError_t launch_split_f32_n3(int map, bool two_d, cudaStream_t st, const KernelArgs &a)
{
    return launch_split_n<float, 3>(map, two_d, st, a);
}
} // namespace rlbmk
