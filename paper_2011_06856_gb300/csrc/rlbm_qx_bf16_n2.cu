// Many-angle quadrant step kernel instances: BF16 storage, N = 2.
#include "rlbm_quad_split.cuh"
namespace rlbmk {
cudaError_t launch_split_bf16_n2(int map, bool two_d, cudaStream_t st, const KernelArgs &a)
{
    return launch_split_n<__nv_bfloat16, 2>(map, two_d, st, a);
}
} // namespace rlbmk
