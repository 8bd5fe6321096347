// Free streaming (tau = infinity) of thin grids, several time steps per launch.
//
// Without a collision the populations do not couple: a step is the bilinear pull of each
// population by itself (Eqs. streaming, interpolation).  One launch per step spent 3.3 us
// on the 2000 x 1, K = 120, N = 3 run of Fig. 2, almost all of it launch and load latency
// (7.7 MB move).  Here a warp owns kCells = 256 consecutive columns of all ny <= 4 rows of
// one population, eight columns a lane in registers, and advances them nsteps <= 32 steps:
// per step one shuffle per row (the neighbour's column) and the interpolation.  The first
// nsteps columns on the upwind side are halo: a column's value at the end depends on
// itself and nsteps columns upwind, so each step spoils one more halo column and the
// others are exact.  Beyond the grid the halo is loaded with the wrapped column (periodic)
// or the edge column (copy-out: the edge column streams from itself, so it and the copies
// stay constant along x in every row).  Every step rounds to the storage type, as single
// steps do.  Columns run through shared memory between coalesced global accesses and the
// lanes' consecutive registers.
#include "rlbm_device.cuh"

namespace rlbmk {

constexpr int kFreeCells = 256; // columns per warp, eight per lane
constexpr int kFreeWarps = 4;
static_assert(kFreeSteps <= kFreeCells / 2, "the halo leaves columns to write");

__device__ __forceinline__ float free_lerp(float a, float to, float from) { return __fmaf_rn(a, __fsub_rn(to, from), from); }
__device__ __forceinline__ double free_lerp(double a, double to, double from) { return __fma_rn(a, __dsub_rn(to, from), from); }

template <class T, int NY>
__global__ void __launch_bounds__(32 * kFreeWarps) rlbm_free_kernel(const KernelArgs a, int N, int pop0, int nsteps)
{
    constexpr int C = kFreeCells / 32, PAD = kFreeCells + kFreeCells / 32;
    __shared__ T buf[kFreeWarps][NY * PAD];
    const int lane = threadIdx.x, w = threadIdx.y;
    const int i = pop0 + blockIdx.y; // population
    const int width = kFreeCells - nsteps, seg = blockIdx.x * kFreeWarps + w;
    if (seg * width >= a.nx) return; // whole warp
    const T *tab = reinterpret_cast<const T *>(a.poptab) + size_t(i) * tab_width(N);
    const T c = __ldg(tab), s = __ldg(tab + 1), ac = fabs(c), as = fabs(s);
    // cell k of the warp is column X(k): downwind from upwind, the first nsteps are halo
    const bool right = c >= T(0); // pulls from x - 1
    const int first = seg * width - nsteps;
    auto X = [&](int k) { return right ? first + k : a.nx - 1 - (first + k); };
    auto slot = [](int k) { return k + (k >> 5); }; // eight consecutive cells per lane without bank conflicts
    const T *fin = reinterpret_cast<const T *>(a.fin) + (long long)i * a.S;
    T *b = buf[w];
#pragma unroll
    for (int j = 0; j < NY; ++j)
#pragma unroll
        for (int m = 0; m < C; ++m) {
            const int k = m * 32 + lane;
            b[j * PAD + slot(k)] = __ldg(fin + (long long)j * a.nx + bc_any(X(k), a.nx, a.bcx));
        }
    __syncwarp();
    T f[NY][C];
#pragma unroll
    for (int j = 0; j < NY; ++j)
#pragma unroll
        for (int m = 0; m < C; ++m) f[j][m] = b[j * PAD + slot(lane * C + m)];
    const bool up = s >= T(0); // pulls from y - 1
    for (int t = 0; t < nsteps; ++t) {
#pragma unroll
        for (int j = 0; j < NY; ++j) {
            const T prev = __shfl_up_sync(0xffffffffu, f[j][C - 1], 1);
#pragma unroll
            for (int m = C - 1; m > 0; --m) f[j][m] = free_lerp(ac, f[j][m - 1], f[j][m]);
            f[j][0] = free_lerp(ac, prev, f[j][0]);
        }
        if constexpr (NY > 1) {
#pragma unroll
            for (int m = 0; m < C; ++m) {
                T h[NY];
#pragma unroll
                for (int j = 0; j < NY; ++j) h[j] = f[j][m];
#pragma unroll
                for (int j = 0; j < NY; ++j) {
                    const T lo = h[j > 0 ? j - 1 : (a.bcy == 0 ? NY - 1 : 0)];
                    const T hi = h[j < NY - 1 ? j + 1 : (a.bcy == 0 ? 0 : NY - 1)];
                    f[j][m] = free_lerp(as, up ? lo : hi, h[j]);
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < NY; ++j)
#pragma unroll
        for (int m = 0; m < C; ++m) b[j * PAD + slot(lane * C + m)] = f[j][m];
    __syncwarp();
    T *fout = reinterpret_cast<T *>(a.fout) + (long long)i * a.S;
#pragma unroll
    for (int j = 0; j < NY; ++j)
#pragma unroll
        for (int m = 0; m < C; ++m) {
            const int k = m * 32 + lane;
            if (k >= nsteps && first + k < a.nx) fout[(long long)j * a.nx + X(k)] = b[j * PAD + slot(k)];
        }
}

cudaError_t launch_free(bool fp64, int N, int first, int count, int nsteps, cudaStream_t st, const KernelArgs &a)
{
    if (nsteps < 1 || nsteps > kFreeSteps || a.ny < 1 || a.ny > kFreeRows || count < 1 || count > kFreePops)
        return cudaErrorInvalidValue;
    void (*k)(const KernelArgs, int, int, int) = nullptr;
    switch (a.ny) {
    case 1: k = fp64 ? rlbm_free_kernel<double, 1> : rlbm_free_kernel<float, 1>; break;
    case 2: k = fp64 ? rlbm_free_kernel<double, 2> : rlbm_free_kernel<float, 2>; break;
    case 3: k = fp64 ? rlbm_free_kernel<double, 3> : rlbm_free_kernel<float, 3>; break;
    default: k = fp64 ? rlbm_free_kernel<double, 4> : rlbm_free_kernel<float, 4>; break;
    }
    const int width = kFreeCells - nsteps, segs = (a.nx + width - 1) / width;
    k<<<dim3((segs + kFreeWarps - 1) / kFreeWarps, count), dim3(32, kFreeWarps), 0, st>>>(a, N, first, nsteps);
    return cudaGetLastError();
}

} // namespace rlbmk
