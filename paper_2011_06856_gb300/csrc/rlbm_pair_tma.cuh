// Tile-staged form of the two-sites-per-lane step (arXiv 2011.06856, Sec. 2.2).
//
// The arithmetic is that of rlbm_quad_kernel (populations in quadruples of
// directions, two sites per lane as packed f32x2 pairs, the per-site part in steps
// shared by the warps); what changes is how the populations reach the registers.  A CTA owns one 64-site tile.  At
// its start the lanes of warp 0 issue the TMA loads of the whole tile into
// shared memory -- cp.async.bulk.tensor over the 3D map {nx, ny, npop}:
//   centre rows  row y of every population, x0 - HX .. x0 + 64 + HX
//                (HX = 16 bytes of halo on each side), CB populations per box;
//   pull rows    (2D) row y - sgn(v_y) of every population (the upwind row of
//                the bilinear pull, Eqs. streaming, interpolation), DB
//                populations per box; the host groups the populations in
//                chunks of DB that share sgn(v_y) (populations with v_y = 0
//                give the pull row the weight 0 and join either side), so one
//                box fetches the right row for a whole chunk;
// and one mbarrier counts the bytes.  While the copies fly, every thread
// copies the quad table into shared memory.  After a bounded
// wait the first pass reads shared memory only, with compile-time offsets; on
// the domain edges the halo cells outside the grid (zero-filled by the TMA)
// are first rewritten with their periodic / copy-out source values.  Several
// CTAs per SM overlap one another's loads, per-site solve and stores.
//
// Stores round stochastically: 16-bit ones with the cvt.rs instruction, FP32
// ones from the FMA residual (quad_relax_sr); random bits from QuadBits
// (rlbm_bits.cuh).
//
// One tile per CTA measured faster than persistent CTAs cycling their tiles
// through one or two stages (every population on its own, three CTAs per SM: 1.44 ms
// against 1.61 ms with one stage and 1.89 ms with two per 2048^2 FP16 step; with four CTAs
// per SM 1.27, with quadruples of directions 0.91).
//
// Every wait is bounded: on expiry the CTA sets bit 1 of the status word,
// waits (again bounded) for its copies and returns without storing.
#pragma once

#include "rlbm_quad.cuh"
#include "rlbm_tma.cuh"

namespace rlbmk {

template <class St> struct PairTmaGeom {
    static constexpr int HX = 16 / int(sizeof(St)); // halo columns on each side (16 bytes)
    static constexpr int BW = kPairSites + 2 * HX;  // box width in x (a multiple of 16 bytes)
};

template <class St, int N, int PP, bool TWO_D>
__device__ __forceinline__ void pair_tma_body(const PairTmaArgs &ta)
{
    constexpr int NC = 2 * N + 1;
    constexpr int QW = PP / 4; // quads per warp
    constexpr int HX = PairTmaGeom<St>::HX, BW = PairTmaGeom<St>::BW;
    constexpr int RW = TWO_D ? 2 : 1;
    const KernelArgs &a = ta.a;
    extern __shared__ __align__(16) unsigned char smem_pt[];
    // TMA destinations: align the base to 1 KB (the host adds the slack)
    unsigned char *sm = smem_pt + ((1024u - (smem_u32(smem_pt) & 1023u)) & 1023u);
    const PairTmaLayout &L = ta.layout;
    const int lane = threadIdx.x, q = threadIdx.y, Gs = blockDim.y, r = threadIdx.z;
    const int g = r * Gs + q, G = Gs * (N + 1);
    const int tid = g * 32 + lane, nthr = G * 32;
    const int npop = a.K * (N + 1);
    St *stage = reinterpret_cast<St *>(sm + L.stage); // [RW][npop][BW]
    float4 *tab = reinterpret_cast<float4 *>(sm + L.tab);
    float *red = reinterpret_cast<float *>(sm + L.red);   // [5][G][64]
    float *sres = reinterpret_cast<float *>(sm + L.sres); // [pair_site_rows(N)][64]
    unsigned long long *bar = reinterpret_cast<unsigned long long *>(sm + L.bar);
    const int x0 = blockIdx.x * kPairSites, y = blockIdx.y;
    const int ym = TWO_D ? bc_index(y - 1, a.ny, a.bcy) : y;
    const int yp = TWO_D ? bc_index(y + 1, a.ny, a.bcy) : y;

    const unsigned seed = __ldcg(a.ctr); // early: its latency passes behind the copies
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (g == 0) {
        if (lane == 0) mbar_expect_tx(bar, unsigned(RW * npop * BW * int(sizeof(St))) + a.extra_tx);
        __syncwarp();
        const int nops = ta.ncbox + (TWO_D ? ta.npbox : 0);
        for (int o = lane; o < nops; o += 32) {
            if (o < ta.ncbox) {
                const int p0 = o * ta.CB;
                tma_load_3d(stage + size_t(p0) * BW, &ta.cmap, x0 - HX, y, p0, bar);
            } else {
                const int c = o - ta.ncbox, p0 = c * ta.DB;
                const bool up = (ta.chunk_up[c >> 6] >> (c & 63)) & 1ull;
                tma_load_3d(stage + size_t(npop + p0) * BW, &ta.pmap, x0 - HX, up ? ym : yp, p0, bar);
            }
        }
    }
    // while the copies fly: the quad table into shared memory
    {
        const float4 *gt = reinterpret_cast<const float4 *>(a.quadtab);
        for (int e = tid; e < (npop >> 2) * 3; e += nthr) tab[e] = __ldg(gt + e);
    }
    const bool arrived = mbar_wait_bounded(bar, 0, a.wait_cycles);
    if (__syncthreads_or(!arrived)) {
        if (tid == 0) {
            atomicOr(a.status, 2);
            mbar_wait_bounded(bar, 0, a.wait_cycles); // the copies still in flight (bounded)
        }
        return;
    }
    const St *fin = reinterpret_cast<const St *>(a.fin);
    const long long S = a.S;
    // halo cells beyond the grid edge (TMA filled zeros): their source values
    const bool left = x0 == 0, right = a.nx - x0 < kPairSites + HX;
    if (left || right) {
        const int xr = a.nx - x0 + HX; // local column of x = nx
        for (int e = tid; e < RW * npop * 2; e += nthr) {
            const int side = e & 1, rest = e >> 1;
            const int rr = rest / npop, p = rest % npop;
            if (side == 0 ? !left : !right) continue;
            int row = y;
            if (rr == 1) {
                const int c = p / ta.DB;
                row = ((ta.chunk_up[c >> 6] >> (c & 63)) & 1ull) ? ym : yp;
            }
            const int xs = bc_index(side == 0 ? -1 : a.nx, a.nx, a.bcx);
            stage[(size_t(rr) * npop + p) * BW + (side == 0 ? HX - 1 : xr)] =
                fin[(long long)p * S + (long long)row * a.nx + xs];
        }
        __syncthreads();
    }

    const int xl = x0 + 2 * lane;
    const bool act = xl < a.nx;
    const int K4 = a.K >> 2, i0 = r * a.K + q * QW; // population a = 0 of the warp's first quad
    const St *cb = stage + size_t(i0) * BW + HX + 2 * lane;        // centre row, this lane's pair
    const St *pb = stage + size_t(npop + i0) * BW + HX + 2 * lane; // pull row
    const int aw = K4 * BW;                                        // to the quad's next population
    const float4 *tb = tab + size_t(r * K4 + q * QW) * 3;

    // pass 1: bilinear pull from shared memory, harmonic sums
    float2 fs[PP];
    QuadSums sums = quad_sums_zero();
#pragma unroll
    for (int k = 0; k < QW; ++k) {
        const float4 t0 = tb[3 * k], t1 = tb[3 * k + 1];
        const float2 c = f2(t0.x, t0.y), sn = f2(t0.z, t0.w);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool left = u == 0 || u == 3; // pulls from x - 1
            const float2 ax = (u & 1) ? sn : c, ay = (u & 1) ? c : sn;
            const St *ra = cb + u * aw + k * BW;
            const float2 C = lds2<St>(ra);
            const float e = lds1<St>(ra + (left ? -1 : 2));
            float2 v = left ? lerp_x<true>(C, e, ax) : lerp_x<false>(C, e, ax);
            if (TWO_D) {
                const St *rb = pb + u * aw + k * BW;
                const float2 C2 = lds2<St>(rb);
                const float e2 = lds1<St>(rb + (left ? -1 : 2));
                const float2 h = left ? lerp_x<true>(C2, e2, ax) : lerp_x<false>(C2, e2, ax);
                v = pfma(ay, psub(h, v), v);
            }
            fs[4 * k + u] = v;
        }
        sums.add(t0, t1, fs + 4 * k);
    }
    if (L.alias) __syncthreads(); // red and sres alias the stage: every warp is done reading it
    sums.store(reinterpret_cast<float2 *>(red), G, g, lane);
    constexpr bool DD = sizeof(St) == 4; // FP32 storage: FP64-class per-site part
    quad_site<N, DD, false>(a, red, G, Gs, G, g, lane, blockIdx.x + blockIdx.y, sres,
                            [&](int s) { return x0 + s < a.nx ? (long long)s : -1ll; });

    // pass 2: this warp's shell coefficients, f^eq, relaxation (Eq. discrete-rbe), stores
    float2 cf[NC], o[3];
    quad_shell<N, DD>(a, r, r, q, Gs, sres, red, lane, cf, o);
    QuadBits rng = quad_seed(unsigned(y) * unsigned(a.nx) + unsigned(xl), unsigned(g), seed);
    const long long Sb = S * (long long)sizeof(St), KS = K4 * Sb;
    char *ob = reinterpret_cast<char *>(a.fout) + i0 * Sb + ((long long)y * a.nx + (act ? xl : 0)) * int(sizeof(St));
#pragma unroll
    for (int k = 0; k < QW; ++k) {
        float2 feq[4], om[4];
        quad_equilibrium<N>(cf, o, tb + 3 * k, feq, om);
        if (k > 0 && 4 * k % QuadBits::kWords == 0) rng.refresh();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            char *p = ob + (k * Sb + u * KS);
            const float2 f = fs[4 * k + u];
            if constexpr (sizeof(St) == 4) {
                const float2 out = quad_relax_sr(f, om[u], feq[u], rng.next());
                if (act) *reinterpret_cast<float2 *>(p) = out;
            } else {
                const unsigned d = cvt2_rs<St>(pfma(om[u], psub(feq[u], f), f), rng.next());
                if (act) *reinterpret_cast<unsigned *>(p) = d;
            }
        }
    }
    __syncthreads();
    if (tid == 0) advance_launch_counter(a.ctr, gridDim.x * gridDim.y);
}

// FP32 storage: the launch bounds of the other two-sites-per-lane kernels.
template <class St, int N, int PP, bool TWO_D>
__global__ void __maxnreg__(PP <= 16 ? 64 : (PP == 24 ? 104 : 128))
    rlbm_pair_tma_kernel(const __grid_constant__ PairTmaArgs ta)
{
    pair_tma_body<St, N, PP, TWO_D>(ta);
}

// 16-bit storage: with PP <= 16, at most 56 registers, so that four CTAs of nine
// warps (the 2048^2 N = 2 K = 48 tiling, 54 KB of shared memory with the aliased
// sums) share an SM.
template <class St, int N, int PP, bool TWO_D>
__global__ void __maxnreg__(PP <= 16 ? 56 : (PP == 24 ? 80 : 96)) rlbm_pair_tma_kernel16(const __grid_constant__ PairTmaArgs ta)
{
    pair_tma_body<St, N, PP, TWO_D>(ta);
}

template <class St, int N, int PP>
static cudaError_t launch_pair_tma_np(bool two_d, dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                      const PairTmaArgs &ta, int *bps)
{
    void (*k)(const PairTmaArgs);
    if constexpr (sizeof(St) == 2)
        k = two_d ? rlbm_pair_tma_kernel16<St, N, PP, true> : rlbm_pair_tma_kernel16<St, N, PP, false>;
    else
        k = two_d ? rlbm_pair_tma_kernel<St, N, PP, true> : rlbm_pair_tma_kernel<St, N, PP, false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (bps) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, k, int(block.x * block.y * block.z), smem);
    k<<<grid, block, smem, st>>>(ta);
    return cudaGetLastError();
}

// The instances of storage St and order N (one compile unit each): one CTA per
// 64-site tile; with bps set, only the occupancy query (CTAs per SM).
template <class St, int N>
static cudaError_t launch_pair_tma_n(int PP, bool two_d, dim3 block, size_t smem, cudaStream_t st,
                                     const PairTmaArgs &ta, int *bps)
{
    const dim3 grid((ta.a.nx + kPairSites - 1) / kPairSites, ta.a.ny);
    switch (PP) {
    case 8: return launch_pair_tma_np<St, N, 8>(two_d, grid, block, smem, st, ta, bps);
    case 12: return launch_pair_tma_np<St, N, 12>(two_d, grid, block, smem, st, ta, bps);
    case 16: return launch_pair_tma_np<St, N, 16>(two_d, grid, block, smem, st, ta, bps);
    case 24: return launch_pair_tma_np<St, N, 24>(two_d, grid, block, smem, st, ta, bps);
    case 32: return launch_pair_tma_np<St, N, 32>(two_d, grid, block, smem, st, ta, bps);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace rlbmk
