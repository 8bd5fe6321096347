// Quadrant form of the FP64-storage step (arXiv 2011.06856, Sec. 2.2; N = 2, 3): the
// populations of a warp in quadruples theta + k pi/2 (rlbm_quad.cuh), one column of the
// grid per lane, RW = 2 rows of it for ny > 1 (P <= 16) or one.  A grid with fewer tiles of
// two rows than the GPU has SMs takes one row: the FP64 pipes of twice the SMs share the work
// (64^2, N = 2, K = 60, P = 12: two rows 59.8 us a step, the per-tile kernel 47.6, one row
// 35.8).
//
// The step is bound by the FP64 pipe (1/64 of the FP32 rate), so what counts is FP64
// operations per population, N = 3 in 2D: the bilinear pull 5 with two rows per lane (the
// interpolation along x of the middle row serves both) or 6, the angular sums 3.25 (5),
// the equilibrium 4 (7), omega 2, relaxation 2: 16.25 against 22 with every population on
// its own.  The per-site part runs once per site, its equilibrium sums in closed form
// (30 operations instead of about 200 with sampled directions), and the shells'
// coefficients once per CTA.
#pragma once

#include "rlbm_device.cuh"

namespace rlbmk {

template <int N, int PP, int RW, bool TWO_D>
__global__ void __maxnreg__(128) rlbm_quad64_kernel(const KernelArgs a)
{
    static_assert(N == 2 || N == 3, "closed forms written for N = 2, 3");
    static_assert(RW == 1 || TWO_D, "two rows per lane need ny > 1");
    constexpr int QW = PP / 4, W = (N + 1) * (N + 1), NC = 2 * N + 1, ST = 32 * RW, TQ = 6;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x, q = threadIdx.y, Gs = blockDim.y, r = threadIdx.z, K4 = a.K >> 2;
    const int g = r * Gs + q, G = Gs * (N + 1);
    double *red = reinterpret_cast<double *>(smem_raw);                    // [5][G][ST], later the coefficients [N+1][NC][ST]
    double *mom = red + (5 * G > (N + 1) * NC ? 5 * G : (N + 1) * NC) * ST; // [8][ST]
    double *sres = mom + 8 * ST;                                           // [W + 3][ST]
    const double *tb = reinterpret_cast<const double *>(a.quadtab) + size_t(r * K4 + q * QW) * TQ;

    const int xl = blockIdx.x * 32 + lane, x = min(xl, a.nx - 1);
    const int y = blockIdx.y * RW;
    const int yb = RW == 2 ? (y + 1 < a.ny ? y + 1 : bc_index(a.ny, a.ny, a.bcy)) : y;
    const int yu = TWO_D ? bc_index(y - 1, a.ny, a.bcy) : y;
    const int yd = TWO_D ? (RW == 2 ? bc_any(y + 2, a.ny, a.bcy) : bc_index(y + 1, a.ny, a.bcy)) : y;
    const int em = bc_index(x - 1, a.nx, a.bcx) - x, ep = bc_index(x + 1, a.nx, a.bcx) - x;
    const long long S = a.S, KS = K4 * S, i0S = (long long)(r * a.K + q * QW) * S;
    const double *fin = reinterpret_cast<const double *>(a.fin) + i0S;
    const double *pa = fin + (long long)y * a.nx + x, *pb = fin + (long long)yb * a.nx + x;
    const double *pu = fin + (long long)yu * a.nx + x, *pd = fin + (long long)yd * a.nx + x;

    double fs[PP][RW];
    double s0[RW], sc[RW], ss[RW], c2[RW], s2[RW];
#pragma unroll
    for (int w = 0; w < RW; ++w) s0[w] = sc[w] = ss[w] = c2[w] = s2[w] = 0.0;
#pragma unroll
    for (int k = 0; k < QW; ++k) {
        double C[4][RW], B[4][RW], D[4], E[4]; // rows of the sites, and the pull row, with their neighbours
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long off = k * S + u * KS;
            const int e = (u == 0 || u == 3) ? em : ep;
            C[u][0] = __ldg(pa + off);
            B[u][0] = __ldg(pa + off + e);
            if constexpr (RW == 2) {
                C[u][1] = __ldg(pb + off);
                B[u][1] = __ldg(pb + off + e);
            }
            if (TWO_D) {
                const double *p = (u < 2 ? pu : pd) + off;
                D[u] = __ldg(p);
                E[u] = __ldg(p + e);
            }
        }
        const double2 cs = __ldg(reinterpret_cast<const double2 *>(tb + TQ * k));
        const double2 cs2 = __ldg(reinterpret_cast<const double2 *>(tb + TQ * k) + 1);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const double ax = (u & 1) ? cs.y : cs.x, ay = (u & 1) ? cs.x : cs.y;
            double v[RW];
#pragma unroll
            for (int w = 0; w < RW; ++w) v[w] = C[u][w] + ax * (B[u][w] - C[u][w]);
            if (TWO_D) {
                const double h = D[u] + ax * (E[u] - D[u]);
                if constexpr (RW == 1) {
                    v[0] += ay * (h - v[0]);
                } else if (u < 2) { // upward: row y pulls from y - 1, row y + 1 from y
                    const double v0 = v[0];
                    v[0] += ay * (h - v0);
                    v[1] += ay * (v0 - v[1]);
                } else {
                    const double v1 = v[1];
                    v[0] += ay * (v1 - v[0]);
                    v[1] += ay * (h - v1);
                }
            }
#pragma unroll
            for (int w = 0; w < RW; ++w) fs[4 * k + u][w] = v[w];
        }
#pragma unroll
        for (int w = 0; w < RW; ++w) {
            const double f0 = fs[4 * k][w], f1 = fs[4 * k + 1][w], f2 = fs[4 * k + 2][w], f3 = fs[4 * k + 3][w];
            const double e02 = f0 + f2, d02 = f0 - f2, e13 = f1 + f3, d13 = f1 - f3, d = e02 - e13;
            s0[w] += e02 + e13;
            sc[w] += cs.x * d02;
            sc[w] -= cs.y * d13;
            ss[w] += cs.y * d02;
            ss[w] += cs.x * d13;
            c2[w] += cs2.x * d;
            s2[w] += cs2.y * d;
        }
    }
#pragma unroll
    for (int w = 0; w < RW; ++w) {
        const int s = w * 32 + lane;
        red[(0 * G + g) * ST + s] = s0[w];
        red[(1 * G + g) * ST + s] = sc[w];
        red[(2 * G + g) * ST + s] = ss[w];
        red[(3 * G + g) * ST + s] = c2[w];
        red[(4 * G + g) * ST + s] = s2[w];
    }
    __syncthreads();
    // the moment folds, one (moment, site) per thread
    const double *sh = reinterpret_cast<const double *>(a.shelltab);
    for (int e = g * 32 + lane; e < 8 * ST; e += G * 32) {
        const int u = e / ST, s = e % ST;
        const double *p = red + (u < 3 ? u : u - 3) * G * ST + s;
        double m = 0.0;
#pragma unroll
        for (int rr = 0; rr <= N; ++rr) {
            double v = p[rr * Gs * ST];
            for (int qq = 1; qq < Gs; ++qq) v += p[(rr * Gs + qq) * ST];
            m += __ldg(sh + 2 * rr + (u < 3 ? 0 : 1)) * v;
        }
        mom[e] = m;
    }
    __syncthreads();
    // the frame and the sums w_{m,k}, one site per thread of RW warps (which rotate with the
    // tile: a fixed choice would keep the same schedulers busy in every resident CTA)
    const int b0 = int((blockIdx.x + blockIdx.y) & 3u) <= G - RW ? int((blockIdx.x + blockIdx.y) & 3u) : 0;
    if (g >= b0 && g < b0 + RW) {
        const int s = (g - b0) * 32 + lane;
        double m[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) m[u] = mom[u * ST + s];
        m[6] = 0.5 * (m[3] + m[6]); // T^xx = (T^tt + C2) / 2, T^xy = S2 / 2
        m[7] = 0.5 * m[7];
        double n, eps, U0, Ux, Uy;
        const bool ok = landau_fast<double>(m, n, eps, U0, Ux, Uy);
        if (!ok && xl < a.nx && y + (g - b0) < a.ny) atomicOr(a.status, 1);
        const double T = eps / (2.0 * n), t1 = n * (N + 1), t2 = t1 * T;
        const double x2 = Ux * Ux, y2 = Uy * Uy, v = x2 + y2, zr = x2 - y2, zi = 2.0 * Ux * Uy;
        const double c = 1.5 * t2 * U0, d = 1.5 * t2;
        auto emit = [&](int row, double w) { sres[row * ST + s] = w; };
        emit(0, t1 / T);
        emit(1, t1 * U0);
        emit(2, t2 * (1.0 + 1.5 * v));
        if constexpr (N == 2) {
            emit(3, t1 * Ux);
            emit(4, c * Ux);
            emit(5, d * zr);
            emit(6, t1 * Uy);
            emit(7, c * Uy);
            emit(8, d * zi);
        } else {
            const double t3 = t2 * T, f = t3 * (2.0 + 2.5 * v), gg = 2.5 * t3, h = gg * U0;
            emit(3, t3 * U0 * (1.0 + 2.5 * v));
            emit(4, t1 * Ux);
            emit(5, c * Ux);
            emit(6, f * Ux);
            emit(7, d * zr);
            emit(8, h * zr);
            emit(9, gg * (zr * Ux - zi * Uy));
            emit(10, t1 * Uy);
            emit(11, c * Uy);
            emit(12, f * Uy);
            emit(13, d * zi);
            emit(14, h * zi);
            emit(15, gg * (zr * Uy + zi * Ux));
        }
        emit(W, U0 * a.inv_tau);
        emit(W + 1, Ux * a.inv_tau);
        emit(W + 2, Uy * a.inv_tau);
    }
    __syncthreads();
    // the Fourier coefficients of every shell (weights folded in): warp q of shell r forms
    // those with index j = q mod Gs, into the angular sums' space
    double *cfs = red + r * NC * ST;
    int turn = q;
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        if (turn == 0) {
            const int m = (j + 1) >> 1;
            int row = 0;
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (i < m) row += N + 1 - i;
            if (j > 0 && !(j & 1)) row += (N + 1) * (N + 2) / 2 - (N + 1);
#pragma unroll
            for (int w = 0; w < RW; ++w) {
                double v = 0.0;
#pragma unroll
                for (int k = 0; k <= N; ++k)
                    if (k >= m) v += a.rqd[(r * (N + 1) + m) * (N + 1) + k] * sres[(row + k - m) * ST + w * 32 + lane];
                cfs[j * ST + w * 32 + lane] = v;
            }
        }
        turn = turn == 0 ? Gs - 1 : turn - 1;
    }
    __syncthreads();
    double *oa = reinterpret_cast<double *>(a.fout) + i0S + (long long)y * a.nx + x;
    const bool act[2] = {xl < a.nx, RW == 2 && xl < a.nx && y + 1 < a.ny};
#pragma unroll
    for (int w = 0; w < RW; ++w) {
        double cf[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) cf[j] = cfs[j * ST + w * 32 + lane];
        const double o0 = sres[W * ST + w * 32 + lane], o1 = sres[(W + 1) * ST + w * 32 + lane];
        const double o2 = sres[(W + 2) * ST + w * 32 + lane];
#pragma unroll
        for (int k = 0; k < QW; ++k) {
            const double2 cs = __ldg(reinterpret_cast<const double2 *>(tb + TQ * k));
            const double2 cs2 = __ldg(reinterpret_cast<const double2 *>(tb + TQ * k) + 1);
            const double h = cf[3] * cs2.x + cf[4] * cs2.y;
            double a0 = cf[1] * cs.x + cf[2] * cs.y, a1 = cf[2] * cs.x - cf[1] * cs.y;
            if constexpr (N == 3) {
                const double2 cs3 = __ldg(reinterpret_cast<const double2 *>(tb + TQ * k) + 2);
                a0 += cf[5] * cs3.x;
                a0 += cf[6] * cs3.y;
                a1 += cf[5] * cs3.y;
                a1 -= cf[6] * cs3.x;
            }
            const double e0 = cf[0] + h, e1 = cf[0] - h;
            const double q0 = o1 * cs.x + o2 * cs.y, q1 = o2 * cs.x - o1 * cs.y;
            const double feq[4] = {e0 + a0, e1 + a1, e0 - a0, e1 - a1};
            const double om[4] = {o0 - q0, o0 - q1, o0 + q0, o0 + q1};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const double f = fs[4 * k + u][w];
                if (act[w]) oa[k * S + u * KS + (w ? a.nx : 0)] = f + om[u] * (feq[u] - f);
            }
        }
    }
}

template <int N, int PP>
static cudaError_t launch_quad64_np(bool one_row, dim3 block, cudaStream_t st, const KernelArgs &a)
{
    void (*k)(const KernelArgs) = a.ny == 1 ? rlbm_quad64_kernel<N, PP, 1, false> : rlbm_quad64_kernel<N, PP, 1, true>;
    int rw = 1;
    if constexpr (PP <= 16) {
        if (a.ny > 1 && !one_row) {
            k = rlbm_quad64_kernel<N, PP, 2, true>;
            rw = 2;
        }
    }
    const int G = int(block.y * block.z), sums = 5 * G, coef = (N + 1) * (2 * N + 1);
    const size_t smem = size_t((sums > coef ? sums : coef) + 8 + (N + 1) * (N + 1) + 3) * 32 * rw * 8;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<dim3((a.nx + 31) / 32, (a.ny + rw - 1) / rw), block, smem, st>>>(a);
    return cudaGetLastError();
}

template <int N>
static cudaError_t launch_quad64_n(int PP, bool one_row, dim3 block, cudaStream_t st, const KernelArgs &a)
{
    switch (PP) {
    case 8: return launch_quad64_np<N, 8>(one_row, block, st, a);
    case 12: return launch_quad64_np<N, 12>(one_row, block, st, a);
    case 16: return launch_quad64_np<N, 16>(one_row, block, st, a);
    case 24: return launch_quad64_np<N, 24>(one_row, block, st, a);
    case 32: return launch_quad64_np<N, 32>(one_row, block, st, a);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace rlbmk
