// Quadrant step kernel instances with the quantum statistics: FP32 storage, N = 3.
#include "rlbm_quad.cuh"
namespace rlbmk {
cudaError_t launch_quad_stat_f32_n3(int PP, int map, bool two_d, dim3 block, size_t smem, cudaStream_t st,
                                    const KernelArgs &a)
{
    return launch_quad_n<float, 3, true>(PP, map, two_d, block, smem, st, a);
}
} // namespace rlbmk
