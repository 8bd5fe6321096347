// Quadrant step kernel for many angles: two passes over the populations of a tile, in one
// launch (K beyond what the warps of a CTA hold in registers; arXiv 2011.06856 Sec. 3 runs
// K = 600, N = 3: 2400 populations, 614 KB for 64 sites).
//
// The moments of a site need all its populations before the first is relaxed.  Parking f*
// on the way makes the CTAs of a tile wait for each other and for the serial per-site part,
// with the SM full of parked values and little to run meanwhile (f* in the shared memory of
// clusters of eight CTAs, 256^2, N = 3, K = 600: 606 us a step, 250 of them independent of K;
// f* in the output buffer, several groups of populations per warp: 660).  Here a pass A
// CTA streams its share of a tile's quads and keeps only the five angular sums; the
// tile's last CTA to arrive does the per-site part (rlbm_quad.cuh, steps A to D) and
// leaves the shells' coefficients in a ring in global memory; a pass B CTA streams the
// same quads again, lag tiles later, and relaxes them.  Nobody waits and any CTA can run
// next to any other: 490 us (2.45 instructions a cycle and SM against 1.5), 1000^2 9.8 to
// 7.3 ms; with the residual of the FP32 stores 505 us and 7.6 ms.  The price is the second read and pull, about a third of the arithmetic; it
// comes from the L2 while lag tiles fit there (K up to about 250).
//
// CTAs are small (four warps, five per SM, 96 registers): a CTA's start and end (ticket,
// first loads, the wait, the counters) cost about as much as three quads per warp.  Eight
// warps x 3 with 80 registers: 557 us, x 2 with 128: 557, four x 6 with 80: 530, x 4 with
// 128: 509, two x 10: 500.
//
// Order.  CTAs take tickets; ticket by ticket the work is A of tile i + lag next to B of
// tile i.  A CTA only waits for work with smaller tickets (B: its tile's coefficients; A:
// that the tile which had its ring place before is done, a ring of 3 lag tiles back), which running
// or finished CTAs hold, so every wait ends.  Waits are bounded all the same: on expiry the
// CTA sets status bit 1 and the abort word, every later CTA returns at once, and the
// launch's last CTA clears the counters.
//
// A tile's counter goes up by PARTS (sums stored), 1 (coefficients stored) and PARTS
// (coefficients read) per launch, PARTS = (N + 1) split_cs; its base value is the launch
// epoch times that, so nothing has to be cleared between launches.
#pragma once

#include "rlbm_quad.cuh"

namespace rlbmk {

__device__ __forceinline__ unsigned split_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// One thread: waits until *word has gone up by at least count since base.  False when the
// wait ran out or another CTA's did.
__device__ __forceinline__ bool split_wait(const KernelArgs &a, const unsigned *word, unsigned base, unsigned count)
{
    const long long t0 = clock64();
    while (split_acquire(word) - base < count) {
        if (*reinterpret_cast<volatile unsigned *>(a.split_sync + 3)) return false;
        if (clock64() - t0 > a.wait_cycles) {
            atomicOr(a.status, 2);
            atomicExch(a.split_sync + 3, 1u);
            return false;
        }
        __nanosleep(100);
    }
    return true;
}

template <class St, int N, int MAP, bool TWO_D>
__global__ void __launch_bounds__(kSplitWarps * 32, kSplitCtasPerSm) rlbm_quad_split_kernel(const KernelArgs a, int ntx, int ntiles)
{
    constexpr int NC = 2 * N + 1, NW = kSplitWarps;
    constexpr bool DD = sizeof(St) == 4;
    using Rows = QuadRows<N, DD>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned s_ticket, s_abort, s_last;
    const int lane = threadIdx.x, q = warp_uniform(threadIdx.y), K4 = a.K >> 2, CS = a.split_cs, PARTS = CS * (N + 1);
    const bool first = q == 0 && lane == 0;
    float *red = reinterpret_cast<float *>(smem_raw); // [5][max(NW, PARTS)][64]
    float *sres = red + 5 * max(NW, PARTS) * kPairSites;

    if (first) {
        s_ticket = atomicAdd(a.split_sync, 1u);
        s_abort = __ldcg(a.split_sync + 3); // one read for the CTA: it may change at any time
    }
    const unsigned seed = __ldcg(a.ctr), base = __ldcg(a.split_sync + 2) * unsigned(2 * PARTS + 1);
    __syncthreads();
    // ticket -> pass, tile, part: A alone for the first lag tiles, B alone for the last
    const int lag = a.split_lag, k = warp_uniform(s_ticket), head = lag * PARTS, mid = (ntiles - lag) * 2 * PARTS;
    bool passB;
    int tile, part;
    if (k < head) {
        passB = false;
        tile = k / PARTS;
        part = k % PARTS;
    } else if (k < head + mid) {
        const int j = k - head, i = j / (2 * PARTS), m = j % (2 * PARTS);
        passB = m & 1;
        tile = passB ? i : i + lag;
        part = m >> 1;
    } else {
        const int j = k - head - mid;
        passB = true;
        tile = ntiles - lag + j / PARTS;
        part = j % PARTS;
    }
    const int r = part / CS, c = part % CS;
    const int j0 = c * K4 / CS + q, j1 = (c + 1) * K4 / CS; // this warp's quads j0, j0 + NW, .. of shell r
    const QuadTile<MAP> t(a, tile % ntx, tile / ntx, lane);
    const float4 *tb = reinterpret_cast<const float4 *>(a.quadtab) + size_t(r) * K4 * 3;
    const long long Sb = a.S * (long long)sizeof(St), KS = K4 * Sb, pop0 = (long long)r * a.K * Sb;
    float *slot = a.split + size_t(tile % a.split_ring) * split_tile_floats(N, CS);
    float *coef = slot + 5 * PARTS * kPairSites, *oslot = coef + (N + 1) * NC * kPairSites;
    unsigned *word = a.split_sync + kSplitSyncWords + tile;

    if (s_abort) {
        // a wait ran out: the step is void and reported
    } else if (!passB) {
        QuadSums sums = quad_sums_zero();
        auto passA = [&](auto edge_tag) {
            using Pull = QuadPull<St, MAP, TWO_D, decltype(edge_tag)::value>;
            const Pull p(a, t, reinterpret_cast<const char *>(a.fin) + pop0);
            typename Pull::Half b[2][2]; // the loads run a quad ahead of the arithmetic
            auto load = [&](int v, int j) {
                if (j >= j1) return;
                p.template load<0>(b[v][0], j * Sb, KS);
                p.template load<1>(b[v][1], j * Sb, KS);
            };
            auto add = [&](int v, int j) {
                if (j >= j1) return;
                const float4 t0 = __ldg(tb + 3 * j), t1 = __ldg(tb + 3 * j + 1);
                float2 f[4];
                Pull::template pull<0>(b[v][0], t0, f);
                Pull::template pull<1>(b[v][1], t0, f);
                sums.add(t0, t1, f);
            };
            load(0, j0);
#pragma unroll 1
            for (int j = j0; j < j1; j += 2 * NW) {
                load(1, j + NW);
                add(0, j);
                load(0, j + 2 * NW);
                add(1, j + NW);
            }
        };
        if (t.interior(a)) passA(QuadTag<false>{});
        else passA(QuadTag<true>{});
        sums.store(reinterpret_cast<float2 *>(red), NW, q, lane);
        // the ring place is free once its former tile's coefficients have been read
        if (first)
            s_last = tile < a.split_ring || split_wait(a, word - a.split_ring, base, unsigned(2 * PARTS + 1)) ? 0u : 2u;
        __syncthreads();
        bool go = s_last == 0u;
        if (go) {
            for (int e = q * 32 + lane; e < 5 * kPairSites; e += NW * 32) {
                const int u = e / kPairSites, s = e % kPairSites;
                const float *p = red + u * NW * kPairSites + s;
                float v = p[0];
#pragma unroll
                for (int w = 1; w < NW; ++w) v += p[w * kPairSites];
                __stcg(slot + (u * PARTS + part) * kPairSites + s, v);
            }
            __threadfence();
        }
        __syncthreads();
        if (first && go) {
            __threadfence();
            s_last = atomicAdd(word, 1u) - base == unsigned(PARTS - 1) ? 1u : 0u;
            __threadfence();
        }
        __syncthreads();
        if (go && s_last == 1u) { // the tile's sums are complete
            for (int e = q * 32 + lane; e < 5 * PARTS * (kPairSites / 4); e += NW * 32)
                reinterpret_cast<float4 *>(red)[e] = __ldcg(reinterpret_cast<const float4 *>(slot) + e);
            quad_site<N, DD, false>(a, red, PARTS, CS, NW, q, lane, unsigned(tile), sres,
                                    [&](int s) { return t.site(a, s); });
            const float2 *w2 = reinterpret_cast<const float2 *>(sres) + lane;
            for (int e = q; e < (N + 1) * NC; e += NW)
                __stcg(reinterpret_cast<float2 *>(coef + e * kPairSites) + lane, quad_coefficient<N, DD>(a, e / NC, w2, e % NC));
            for (int u = q; u < 3; u += NW) __stcg(reinterpret_cast<float2 *>(oslot + u * kPairSites) + lane, w2[(Rows::O + u) * 32]);
            __threadfence();
            __syncthreads();
            if (first) {
                __threadfence();
                atomicAdd(word, 1u);
            }
        }
    } else {
        QuadBits rng = quad_seed(unsigned(t.y) * unsigned(a.nx) + unsigned(t.x), unsigned(part * NW + q), seed);
        const QuadOut<St, MAP> out(a, t, reinterpret_cast<char *>(a.fout) + pop0);
        auto passB_run = [&](auto edge_tag) {
            using Pull = QuadPull<St, MAP, TWO_D, decltype(edge_tag)::value>;
            const Pull p(a, t, reinterpret_cast<const char *>(a.fin) + pop0);
            typename Pull::Half b[2];
            auto load = [&](int j) {
                if (j >= j1) return;
                p.template load<0>(b[0], j * Sb, KS);
                p.template load<1>(b[1], j * Sb, KS);
            };
            load(j0); // before the wait
            if (first) s_last = split_wait(a, word, base, unsigned(PARTS + 1) + (a.extra_tx << 16)) ? 0u : 2u;
            __syncthreads();
            if (s_last) return;
            float2 cf[NC], o[3];
#pragma unroll
            for (int j = 0; j < NC; ++j) cf[j] = __ldcg(reinterpret_cast<const float2 *>(coef + (r * NC + j) * kPairSites) + lane);
#pragma unroll
            for (int u = 0; u < 3; ++u) o[u] = __ldcg(reinterpret_cast<const float2 *>(oslot + u * kPairSites) + lane);
#pragma unroll 1
            for (int j = j0; j < j1; j += NW) {
                const float4 tq[3] = {__ldg(tb + 3 * j), __ldg(tb + 3 * j + 1),
                                      N == 3 ? __ldg(tb + 3 * j + 2) : make_float4(0.f, 0.f, 0.f, 0.f)};
                float2 f[4], feq[4], om[4];
                Pull::template pull<0>(b[0], tq[0], f);
                Pull::template pull<1>(b[1], tq[0], f);
                load(j + NW); // its latency passes behind the equilibrium and the stores
                quad_equilibrium<N>(cf, o, tq, feq, om);
                out.store(j * Sb, KS, f, feq, om, rng);
                constexpr int TURN = (QuadBits::kWords / 4 - 1) * NW; // the warp's fourth quad since the last one
                static_assert((NW & (NW - 1)) == 0, "quads counted by the bits of j - j0");
                if (((j - j0) & TURN) == TURN) rng.refresh();
            }
        };
        if (t.interior(a)) passB_run(QuadTag<false>{});
        else passB_run(QuadTag<true>{});
        __syncthreads(); // every warp has read the coefficients
        if (first && s_last == 0u) {
            __threadfence();
            atomicAdd(word, 1u);
        }
    }
    // the launch's last CTA: the next epoch and the launch counter
    __syncthreads();
    if (first) {
        __threadfence();
        if (atomicAdd(a.split_sync + 1, 1u) == gridDim.x - 1) {
            a.split_sync[0] = 0u;
            a.split_sync[1] = 0u;
            if (*reinterpret_cast<volatile unsigned *>(a.split_sync + 3)) { // start over
                for (int i = 0; i < ntiles; ++i) a.split_sync[kSplitSyncWords + i] = 0u;
                a.split_sync[2] = 0u;
                a.split_sync[3] = 0u;
            } else {
                a.split_sync[2] += 1u;
            }
            __threadfence();
            atomicAdd(a.ctr, 1u);
        }
    }
}

template <class St, int N>
static cudaError_t launch_split_n(int map, bool two_d, cudaStream_t st, const KernelArgs &a)
{
    void (*k)(const KernelArgs, int, int);
    int ntx = (a.nx + 63) / 64, nty = a.ny;
    switch (map) {
    case kMapRow: k = two_d ? rlbm_quad_split_kernel<St, N, kMapRow, true> : rlbm_quad_split_kernel<St, N, kMapRow, false>; break;
    case kMapCol:
        k = rlbm_quad_split_kernel<St, N, kMapCol, true>;
        ntx = (a.nx + 31) / 32;
        nty = (a.ny + 1) / 2;
        break;
    case kMapSplit: k = rlbm_quad_split_kernel<St, N, kMapSplit, false>; break;
    default: return cudaErrorInvalidValue;
    }
    const int parts = a.split_cs * (N + 1), ntiles = ntx * nty;
    KernelArgs b = a;
    b.split_lag = a.split_lag < ntiles ? a.split_lag : ntiles;
    const size_t smem = size_t(5 * (parts > kSplitWarps ? parts : kSplitWarps) + pair_site_rows(N)) * kPairSites * 4;
    k<<<2 * parts * ntiles, dim3(32, kSplitWarps), smem, st>>>(b, ntx, ntiles);
    return cudaGetLastError();
}

} // namespace rlbmk
