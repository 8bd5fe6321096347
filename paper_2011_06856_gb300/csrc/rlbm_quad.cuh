// Quadrant form of the two-sites-per-lane arithmetic (arXiv 2011.06856, Sec. 2.2).
//
// With K a multiple of 4 the angles of a shell come in quadruples: theta, theta +
// pi/2, theta + pi, theta + 3 pi/2 (populations j, j + K/4, j + K/2, j + 3 K/4 of the
// shell, j < K/4, 0 <= theta < pi/2), with directions (c, s), (-s, c), (-c, -s),
// (s, -c).  A warp owns whole quadruples ("quads"), which
//  - fixes the pull directions at compile time: population a of a quad comes from
//    (x - 1, y - 1), (x + 1, y - 1), (x + 1, y + 1), (x - 1, y + 1) with the weights
//    (c, s) for a = 0, 2 and (s, c) for a = 1, 3: no sign masks, no selects, no |v|;
//  - shares the angular sums: with e02 = f0 + f2, d02 = f0 - f2 (likewise e13, d13),
//    S0 += e02 + e13, Sc += c d02 - s d13, Ss += s d02 + c d13 (the signs in a second accumulator),
//    C2 += cos 2t (e02 - e13), S2 += sin 2t (e02 - e13): 13 operations for four
//    populations instead of 24;
//  - shares the equilibrium: the harmonics of even order agree on opposite
//    directions and change sign by quarter turns, those of odd order the other way
//    round: 12 (N = 2) or 16 (N = 3) operations for four populations instead of 28
//    or 44, and omega = (U^0 - U.v) / tau needs 8 instead of 8 with no table of its own;
//  - needs one table entry per quad: (c,c,s,s), (cos 2t, cos 2t, sin 2t, sin 2t) and
//    for N = 3 the third harmonic.
// The weights w_i of a shell are equal, so they are folded into its projection weights
// (KernelArgs::rq).
//
// The per-site part uses closed forms: the moments of the boosted rest-frame direction
// q on the light cone are
//    < (q^0)^(k-m) (q^x + i q^y)^m > = (k-m)!/k! P_k^(m)(U^0) (U^x + i U^y)^m
// (P_k^(m): m-th derivative of the Legendre polynomial; Laplace's integral), written in
// v = Ux^2 + Uy^2 = (U^0)^2 - 1, in which every coefficient is positive: no
// cancellation.  They replace the sum over N + 1 sampled directions (about 2000 of the
// 3400 FP32 instructions per site of the double-float solve for N = 3).
#pragma once

#include "rlbm_pair.cuh"

#include <type_traits>

namespace rlbmk {

// ---- the per-site part, for the tile's 64 sites ------------------------------------
//
// Its serial chain, not its instruction count, held a tile back when two warps did it
// whole (about 1900 dependent-heavy instructions for FP32 storage, N = 3): it is cut into
// steps that all warps share, with a CTA barrier after each:
//   A  one warp per moment, two sites a lane: the moment fold, compensated for FP32 storage;
//   B  one thread per site, two warps: the Landau frame, t_k = (N + 1) n T^(k-1);
//   C  (FP32 storage) one warp per group of rows: the sums w_{m,k} of two sites a lane;
//      16-bit storage forms them in step B;
//   D  the warps of a shell: its Fourier coefficients (quad_shell).
// The two warps of step B rotate with the tile: a fixed choice would put the chains of
// all resident CTAs on the same two of the SM's four schedulers.
//
// Rows of 64 floats in shared memory: red [5 G], the warps' harmonic sums, dead after A;
// then U (hi, lo) and t_1..t_N (hi, lo) in its first rows, the coefficients of step D
// after them.  sres: row 0 (and W, lo) t_0; the moments in rows that B does not write;
// after C the sums w_{m,k}, hi rows, lo rows; U^a / tau in the three rows after them.
template <int N, bool DD> struct QuadRows {
    static constexpr int W = (N + 1) * (N + 1);
    static constexpr int O = DD ? 2 * W : W;             // U^a / tau
    static constexpr int FRAME = DD ? 2 * (3 + N) : 0;   // rows of red kept for the frame
    // row of moment u (hi), and for FP32 storage of its low part: rows 1.. of sres
    // skipping W, which holds the low part of t_0
    static __device__ __forceinline__ int mom(int u) { return u + 1 + (DD && u + 1 >= W ? 1 : 0); }
};

// Step A.  Moments N^t, N^x, N^y, T^tt, T^tx, T^ty, then the C2 and S2 folds for T^xx =
// (T^tt + C2) / 2 and T^xy = S2 / 2: warp g of nw takes moments g,
// g + nw, .., two sites a lane.
template <int N, bool DD>
__device__ __forceinline__ void quad_moments(const KernelArgs &a, const float *red, int G, int Gs, int nw, int g,
                                             int lane, float *sres)
{
    using R = QuadRows<N, DD>;
    float2 *out = reinterpret_cast<float2 *>(sres) + lane;
    for (int u = g; u < 8; u += nw) {
        const float2 *p = reinterpret_cast<const float2 *>(red) + (u < 3 ? u : u - 3) * G * 32 + lane;
        float2 s = f2(0.f, 0.f), e = s;
#pragma unroll
        for (int rr = 0; rr <= N; ++rr) {
            float2 x = *p; // the warps' FP32 sums of one shell, added in FP32
            p += 32;
            for (int qq = 1; qq < Gs; ++qq, p += 32) x = padd(x, *p);
            const float2 f = a.shellq[2 * rr + (u < 3 ? 0 : 1)], fh = f2(f.x, f.x);
            if (!DD) {
                s = pfma(fh, x, s);
                continue;
            }
            // compensated dot product (Ogita, Rump and Oishi, 2005): s + e += (fh + fl) x
            const float2 pr = pmul(fh, x), pe = pfma(fh, x, pneg(pr)); // exact: fh x = pr + pe
            const df2 t = p_two_sum(s, pr);
            s = t.hi;
            e = padd(pfma(f2(f.y, f.y), x, e), padd(pe, t.lo));
        }
        out[R::mom(u) * 32] = s;
        if (DD) out[R::mom(8 + u) * 32] = e;
    }
}

// The quantum statistics' part of step B: from (n, e) the site's (eta, T) and t_k =
// (N + 1) 2 pi g T^(k+1) phi_{k+1}, in FP64 (stat_solve_fd_short: about 150 FP64
// operations; where it declines, and for Bose-Einstein, stat_solve), kept as double-floats.
template <int N>
__device__ __noinline__ bool quad_statistics(const KernelArgs &a, df64 n, df64 e, long long site, df64 *t)
{
    const double nd = double(n.hi) + double(n.lo), ed = double(e.hi) + double(e.lo);
    const double x0 = a.qeta[site];
    double eta, T, phi[6];
    bool ok = true;
    if (!(a.stat > 0 && stat_solve_fd_short(nd, ed, a.gdeg, x0, eta, T, phi)))
        ok = stat_solve(nd, ed, a.gdeg, a.stat, eta, T, x0, phi, N + 1, 1e-5);
    double w = 6.283185307179586477 * (N + 1) * a.gdeg * T;
#pragma unroll
    for (int k = 0; k <= N; ++k) {
        const double v = w * phi[k];
        t[k].hi = float(v);
        t[k].lo = float(v - double(t[k].hi));
        w *= T;
    }
    a.qeta[site] = eta; // the next step's start
    return ok;
}

// Step B for site s, FP32 storage: the frame in double-float; site: its index in the grid
// (act: it lies in it).
template <int N, bool QUANT>
__device__ __forceinline__ void quad_frame_dd(const KernelArgs &a, int s, long long site, bool act, float *sres, float *fr)
{
    using R = QuadRows<N, true>;
    constexpr int ST = kPairSites;
    df64 m[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) m[u] = fast_two_sum(sres[R::mom(u) * ST + s], sres[R::mom(8 + u) * ST + s]);
    m[6] = (m[3] + m[6]) * 0.5f;
    m[7] = m[7] * 0.5f;
    df64 n, eps, U0, Ux, Uy;
    bool ok = landau_dd(m, n, eps, U0, Ux, Uy);
    df64 t[N + 1];
    if constexpr (QUANT) {
        if (act) ok = quad_statistics<N>(a, n, eps, site, t) && ok;
        else
            for (int k = 0; k <= N; ++k) t[k] = dd(1.f);
    } else {
        const df64 T = eps / (n * 2.f);
        t[1] = n * float(N + 1);
        t[0] = t[1] / T;
#pragma unroll
        for (int k = 2; k <= N; ++k) t[k] = t[k - 1] * T;
    }
    if (!ok && act) atomicOr(a.status, 1);
    const df64 f[3] = {U0, Ux, Uy};
#pragma unroll
    for (int u = 0; u < 3; ++u) {
        fr[2 * u * ST + s] = f[u].hi;
        fr[(2 * u + 1) * ST + s] = f[u].lo;
        sres[(R::O + u) * ST + s] = to_float(f[u]) * a.inv_tau_f;
    }
    sres[s] = t[0].hi;
    sres[R::W * ST + s] = t[0].lo;
#pragma unroll
    for (int k = 1; k <= N; ++k) {
        fr[(4 + 2 * k) * ST + s] = t[k].hi;
        fr[(5 + 2 * k) * ST + s] = t[k].lo;
    }
}

// Step B for site s, 16-bit storage: the frame in FP32, refined in double-float where
// T^ab is near-degenerate, and the equilibrium sums (rows as in step C).
template <int N>
__device__ __forceinline__ void quad_frame_f32(const KernelArgs &a, int s, bool act, float *sres)
{
    using R = QuadRows<N, false>;
    constexpr int ST = kPairSites;
    float m[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) m[u] = sres[R::mom(u) * ST + s];
    m[6] = a.off_f[6] + 0.5f * (m[3] + m[6]);
    m[7] = a.off_f[7] + 0.5f * m[7];
#pragma unroll
    for (int u = 0; u < 6; ++u) m[u] += a.off_f[u];
    float n, eps, U0, Ux, Uy;
    const bool ok = landau_f32_adaptive(m, n, eps, U0, Ux, Uy);
    if (!ok && act) atomicOr(a.status, 1);
    const float T = __fdividef(eps, 2.f * n);
    const float t1 = n * float(N + 1), t2 = t1 * T;
    const float x2 = Ux * Ux, y2 = Uy * Uy, v = x2 + y2, zr = x2 - y2, zi = 2.f * Ux * Uy;
    const float c = 1.5f * t2 * U0, d = 1.5f * t2;
    auto emit = [&](int row, float w) { sres[row * ST + s] = w; };
    emit(0, __fdividef(t1, T));
    emit(1, t1 * U0);
    emit(2, t2 * (1.f + 1.5f * v));
    if constexpr (N == 2) {
        emit(3, t1 * Ux);
        emit(4, c * Ux);
        emit(5, d * zr);
        emit(6, t1 * Uy);
        emit(7, c * Uy);
        emit(8, d * zi);
    } else {
        const float t3 = t2 * T, f = t3 * (2.f + 2.5f * v), g = 2.5f * t3, h = g * U0;
        emit(3, t3 * U0 * (1.f + 2.5f * v));
        emit(4, t1 * Ux);
        emit(5, c * Ux);
        emit(6, f * Ux);
        emit(7, d * zr);
        emit(8, h * zr);
        emit(9, g * (zr * Ux - zi * Uy));
        emit(10, t1 * Uy);
        emit(11, c * Uy);
        emit(12, f * Uy);
        emit(13, d * zi);
        emit(14, h * zi);
        emit(15, g * (zr * Uy + zi * Ux));
    }
    sres[(R::O + 0) * ST + s] = U0 * a.inv_tau_f;
    sres[(R::O + 1) * ST + s] = Ux * a.inv_tau_f;
    sres[(R::O + 2) * ST + s] = Uy * a.inv_tau_f;
}

// Step C, FP32 storage: the sums w_{m,k} = t_k <q0^(k-m) z^m> (Re rows m = 0..N, k = m..N,
// then Im rows m = 1..N, k = m..N) in packed double-float, warp g of nw taking groups g, g + nw, ...
template <int N>
__device__ __forceinline__ void quad_sums_dd(const float *fr, int nw, int g, int lane, float *sres)
{
    constexpr int W = (N + 1) * (N + 1), IM = (N + 1) * (N + 2) / 2; // first Im row
    const float2 *f2r = reinterpret_cast<const float2 *>(fr) + lane;
    float2 *out = reinterpret_cast<float2 *>(sres) + lane;
    auto val = [&](int i) { return df2{f2r[2 * i * 32], f2r[(2 * i + 1) * 32]}; }; // U0, Ux, Uy, t_1, ..
    auto emit = [&](int row, df2 w) {
        out[row * 32] = w.hi;
        out[(W + row) * 32] = w.lo;
    };
    constexpr int NG = N == 2 ? 4 : 7;
    for (int task = g; task < NG; task += nw) {
        const df2 U0 = val(0), Ux = val(1), Uy = val(2);
        switch (task) {
        case 0: {
            const df2 t = val(3);
            emit(1, t * U0);
            emit(N + 1, t * Ux);
            emit(IM, t * Uy);
            break;
        }
        case 1: {
            const df2 v = Ux * Ux + Uy * Uy;
            emit(2, val(4) * (v * 1.5f + 1.f));
            if constexpr (N == 3) emit(3, (val(5) * U0) * (v * 2.5f + 1.f));
            break;
        }
        case 2: {
            const df2 t = (val(4) * U0) * 1.5f;
            emit(N + 2, t * Ux);
            emit(IM + 1, t * Uy);
            break;
        }
        case 3: {
            const df2 t = val(4) * 1.5f;
            emit(2 * N + 1, t * (Ux * Ux - Uy * Uy));
            emit(IM + N, t * ((Ux * Uy) * 2.f));
            break;
        }
        default:
            if constexpr (N == 3) {
                const df2 t = val(5) * 2.5f;
                if (task == 4) {
                    const df2 v = Ux * Ux + Uy * Uy, f = val(5) * (v * 2.5f + 2.f);
                    emit(6, f * Ux);
                    emit(12, f * Uy);
                } else {
                    const df2 zr = Ux * Ux - Uy * Uy, zi = (Ux * Uy) * 2.f;
                    if (task == 5) {
                        const df2 f = t * U0;
                        emit(8, f * zr);
                        emit(14, f * zi);
                    } else {
                        emit(9, t * (zr * Ux - zi * Uy));
                        emit(15, t * (zr * Uy + zi * Ux));
                    }
                }
            }
        }
    }
}

// Steps A to C; site(s) gives the grid index of site s of the tile, or -1 outside the
// grid; rot picks the warps of step B.  red holds the sums of G groups of populations, Gs
// per shell; the CTA has nw warps, g is this one.  Every thread of the CTA calls this after
// the sums are stored; it ends with a CTA barrier.
template <int N, bool DD, bool QUANT, class Site>
__device__ __forceinline__ void quad_site(const KernelArgs &a, float *red, int G, int Gs, int nw, int g, int lane,
                                          unsigned rot, float *sres, Site site)
{
    __syncthreads();
    quad_moments<N, DD>(a, red, G, Gs, nw, g, lane, sres);
    __syncthreads();
    const int b0 = int(rot & 3u) < nw - 1 ? int(rot & 3u) : 0; // two neighbouring warps of the first four
    if (g == b0 || g == b0 + 1) {
        const int s = (g - b0) * 32 + lane;
        const long long i = site(s);
        if constexpr (DD) quad_frame_dd<N, QUANT>(a, s, i, i >= 0, sres, red);
        else quad_frame_f32<N>(a, s, i >= 0, sres);
    }
    __syncthreads();
    if constexpr (DD) {
        quad_sums_dd<N>(red, nw, g, lane, sres);
        __syncthreads();
    }
}

// One Fourier coefficient of shell r's equilibrium for the lane's two sites (packed):
// index j = 0: Re C_0 (less the storage offset), 2m - 1, 2m: Re, Im C_m, in stored units
// with the weight of the shell's populations.  DD: the w_{m,k} are double-floats (hi rows,
// then lo rows) and the radial sum is a packed compensated dot product, rounded once.
template <int N, bool DD>
__device__ __forceinline__ float2 quad_coefficient(const KernelArgs &a, int r, const float2 *w2, int j)
{
    constexpr int W = (N + 1) * (N + 1);
    const int m = (j + 1) >> 1;
    int row = 0; // first row of mode m (Re rows, then Im rows)
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (i < m) row += N + 1 - i;
    if (j > 0 && !(j & 1)) row += (N + 1) * (N + 2) / 2 - (N + 1);
    const float2 *rt = a.rq + (r * (N + 1) + m) * (N + 1);
    if constexpr (DD) {
        float2 s = f2(0.f, 0.f), e = s;
#pragma unroll
        for (int k = 0; k <= N; ++k) {
            if (k < m) continue;
            const float2 t = rt[k], th = f2(t.x, t.x);
            const float2 h = w2[(row + k - m) * 32];
            const float2 p = pmul(th, h);
            const float2 pe = pfma(th, h, pneg(p)); // exact: th h = p + pe
            const float2 lo = pfma(th, w2[(W + row + k - m) * 32], pmul(f2(t.y, t.y), h));
            if (k == m) {
                s = p;
                e = padd(pe, lo);
            } else {
                const df2 u = p_two_sum(s, p);
                s = u.hi;
                e = padd(padd(e, lo), padd(pe, u.lo));
            }
        }
        return padd(s, e);
    } else {
        // 16-bit deviation form: f^eq less the rest equilibrium (beta = 1 in stored units)
        float2 out = j == 0 ? f2(-a.beta_f, -a.beta_f) : f2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k <= N; ++k) {
            if (k < m) continue;
            const float t = rt[k].x;
            out = pfma(f2(t, t), w2[(row + k - m) * 32], out);
        }
        return out;
    }
}

// Shell r's 2N + 1 coefficients cf for the lane's two sites, and o = U^a / tau.  The Gs
// warps of a shell need the same coefficients: warp q forms those with index j = q mod
// Gs and they share them through cs (the angular sums' space, after the frame's rows:
// FRAME + (N + 1)(2N + 1) <= 5 G rows for Gs >= 2; slot: the shell's place there); a
// shell's only warp forms them all.  Every thread of the CTA calls this.
template <int N, bool DD>
__device__ __forceinline__ void quad_shell(const KernelArgs &a, int r, int slot, int q, int Gs, const float *sres,
                                           float *cs, int lane, float2 *cf, float2 *o)
{
    using R = QuadRows<N, DD>;
    constexpr int NC = 2 * N + 1, OR = R::O;
    const float2 *w2 = reinterpret_cast<const float2 *>(sres) + lane;
    if (Gs == 1) {
#pragma unroll
        for (int j = 0; j < NC; ++j) cf[j] = quad_coefficient<N, DD>(a, r, w2, j);
    } else {
        float2 *c2 = reinterpret_cast<float2 *>(cs) + (R::FRAME + slot * NC) * 32 + lane;
        int turn = q; // coefficients until this warp's next one
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            if (turn == 0) c2[j * 32] = quad_coefficient<N, DD>(a, r, w2, j);
            turn = turn == 0 ? Gs - 1 : turn - 1;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NC; ++j) cf[j] = c2[j * 32];
    }
#pragma unroll
    for (int u = 0; u < 3; ++u) o[u] = w2[(OR + u) * 32];
}

// The five harmonic sums of a warp's populations, two sites per lane.
struct QuadSums {
    float2 s0, sc, sa, sb, c2, s2; // Ss = sa - sb

    __device__ __forceinline__ void add(float4 t0, float4 t1, const float2 *f)
    {
        const float2 c = f2(t0.x, t0.y), s = f2(t0.z, t0.w);
        const float2 e02 = padd(f[0], f[2]), d02 = psub(f[0], f[2]);
        const float2 e13 = padd(f[1], f[3]), d31 = psub(f[3], f[1]);
        const float2 D = psub(e02, e13);
        s0 = padd(s0, padd(e02, e13));
        sc = pfma(s, d31, pfma(c, d02, sc));
        sa = pfma(s, d02, sa);
        sb = pfma(c, d31, sb);
        c2 = pfma(f2(t1.x, t1.y), D, c2);
        s2 = pfma(f2(t1.z, t1.w), D, s2);
    }
    __device__ __forceinline__ void store(float2 *red2, int G, int g, int lane) const
    {
        red2[(0 * G + g) * 32 + lane] = s0;
        red2[(1 * G + g) * 32 + lane] = sc;
        red2[(2 * G + g) * 32 + lane] = psub(sa, sb);
        red2[(3 * G + g) * 32 + lane] = c2;
        red2[(4 * G + g) * 32 + lane] = s2;
    }
};
__device__ __forceinline__ QuadSums quad_sums_zero()
{
    const float2 z = f2(0.f, 0.f);
    return {z, z, z, z, z, z};
}

// f^eq and omega of a quad's four populations (two sites per lane).
template <int N>
__device__ __forceinline__ void quad_equilibrium(const float2 *cf, const float2 *o, const float4 *t, float2 *feq,
                                                 float2 *om)
{
    const float4 t0 = t[0], t1 = t[1];
    const float2 c = f2(t0.x, t0.y), s = f2(t0.z, t0.w);
    const float2 h = pfma(cf[4], f2(t1.z, t1.w), pmul(cf[3], f2(t1.x, t1.y)));
    // odd part along theta, a0, and along theta + pi/2, a1 - b1
    float2 a0 = pfma(cf[2], s, pmul(cf[1], c)), a1 = pmul(cf[2], c), b1 = pmul(cf[1], s);
    if constexpr (N == 3) {
        const float4 t2 = t[2];
        const float2 c3 = f2(t2.x, t2.y), s3 = f2(t2.z, t2.w);
        a0 = pfma(cf[5], c3, pfma(cf[6], s3, a0));
        a1 = pfma(cf[5], s3, a1);
        b1 = pfma(cf[6], c3, b1);
    }
    a1 = psub(a1, b1);
    const float2 e0 = padd(cf[0], h), e1 = psub(cf[0], h);
    feq[0] = padd(e0, a0);
    feq[2] = psub(e0, a0);
    feq[1] = padd(e1, a1);
    feq[3] = psub(e1, a1);
    const float2 q0 = pfma(o[1], c, pmul(o[2], s)), q1 = psub(pmul(o[2], c), pmul(o[1], s));
    om[0] = psub(o[0], q0);
    om[2] = padd(o[0], q0);
    om[1] = psub(o[0], q1);
    om[3] = padd(o[0], q1);
}

// Bilinear pull of two sites from the streamed rows: C, C2 the centre and pull-row
// pairs, e, e2 their outer neighbours; LEFT: the neighbour is at x - 1 (the pair is
// (e, C.x)), else at x + 2 (the pair is (C.y, e)).  ax, ay: the weights |v_x|, |v_y|.
template <bool LEFT>
__device__ __forceinline__ float2 lerp_x(float2 C, float e, float2 ax)
{
    const float in = LEFT ? C.x - C.y : C.y - C.x; // the difference inside the pair
    const float2 d = LEFT ? f2(e - C.x, in) : f2(in, e - C.y);
    return pfma(ax, d, C);
}

// The relaxation f* + om (f^eq - f*) of two FP32 sites, rounded stochastically.  r, the
// result rounded to nearest, gives the binade; e is what that rounding lost (the FMA's
// residual, exact while |om d| < |f*| / 2); noise uniform in +- ulp(r) / 2 is added to it
// before the last rounding, whose mean is then the unrounded value.  Without e, as f* +
// (om d + noise), om d is first rounded to its own unit: the last rounding meets ties, and
// its mean is off by 0.016 ulp rms at om = 0.3, |d| = f* / 10, by 0.05 to 0.2 ulp beyond (round
// to nearest: 0.29), the same at every step of a steady flow.
__device__ __forceinline__ float2 quad_relax_sr(float2 fs, float2 om, float2 feq, unsigned rb)
{
    const float2 d = psub(feq, fs);
    const float2 r = pfma(om, d, fs);
    const float2 e = pfma(om, d, psub(fs, r));
    // 23 random bits below the exponent of 2^-23, from bit 31 down for one site and from
    // bit 15 down (cyclically) for the other: uniform in 2^-23 [1, 2), less 1.5 2^-23
    const unsigned b0 = __funnelshift_r(rb, 0x68u, 9), b1 = __funnelshift_r(__funnelshift_l(rb, rb, 16), 0x68u, 9);
    const float2 u = padd(f2(__uint_as_float(b0), __uint_as_float(b1)), f2(-1.78813934326171875e-7f, -1.78813934326171875e-7f));
    const float2 two_e = f2(__uint_as_float(__float_as_uint(r.x) & 0x7f800000u),
                            __uint_as_float(__float_as_uint(r.y) & 0x7f800000u));
    return padd(r, pfma(u, two_e, e));
}

// Two 16-bit values with the stochastic-rounding conversion (the first source operand
// lands in the upper half).
template <class St> __device__ __forceinline__ unsigned cvt2_rs(float2 v, unsigned rbits);
template <> __device__ __forceinline__ unsigned cvt2_rs<__half>(float2 v, unsigned rbits)
{
    unsigned d;
    asm("cvt.rs.satfinite.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v.y), "f"(v.x), "r"(rbits));
    return d;
}
template <> __device__ __forceinline__ unsigned cvt2_rs<__nv_bfloat16>(float2 v, unsigned rbits)
{
    unsigned d;
    asm("cvt.rs.satfinite.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(v.y), "f"(v.x), "r"(rbits));
    return d;
}

template <bool B> struct QuadTag {
    static constexpr bool value = B;
};

// v, which is the same in every lane, as a value the compiler knows to be (a shuffle from a
// fixed lane): what follows from it runs on the uniform pipe.
__device__ __forceinline__ int warp_uniform(unsigned v) { return int(__shfl_sync(0xffffffffu, v, 0)); }

// The place of a CTA's 64 sites in the grid.
template <int MAP> struct QuadTile {
    static constexpr bool COL = MAP == kMapCol, SPLIT = MAP == kMapSplit;
    int x0, y, x, x2; // tile corner; the lane's column(s), clamped into the grid
    bool act0, act1;  // the lane's sites lie in the grid
    __device__ __forceinline__ QuadTile(const KernelArgs &a, int bx, int by, int lane)
    {
        x0 = bx * (COL ? 32 : 64);
        y = by * (COL ? 2 : 1);
        const int xl = x0 + (MAP == kMapRow ? 2 * lane : lane);
        x = min(xl, MAP == kMapRow ? a.nx - 2 : a.nx - 1);
        x2 = SPLIT ? min(xl + 32, a.nx - 1) : x; // the lane's second site
        act0 = xl < a.nx;
        act1 = COL ? (act0 && y + 1 < a.ny) : (SPLIT ? xl + 32 < a.nx : act0);
    }
    __device__ __forceinline__ bool interior(const KernelArgs &a) const { return x0 > 0 && x0 + (COL ? 32 : 64) < a.nx; }
    // grid index of site s (lane s / 2's first or second), -1 outside the grid
    __device__ __forceinline__ long long site(const KernelArgs &a, int s) const
    {
        const int xs = x0 + (MAP == kMapRow ? s : (s >> 1) + (SPLIT ? 32 * (s & 1) : 0));
        const int ys = y + (COL ? s & 1 : 0);
        return xs < a.nx && ys < a.ny ? (long long)ys * a.nx + xs : -1ll;
    }
};

// The bilinear pull (Eqs. streaming, interpolation) of half a quad: populations u = H and
// H + 2.  EDGE: the tile touches the x boundary, a lane's neighbours are at its own
// wrapped or clamped offsets; else they are at fixed offsets from the centre.
//
// Addresses: base, the rows and the quad are the same for all lanes of a warp, so a
// population's row is a uniform 64-bit address (formed on the uniform pipe) and a lane adds
// its 32-bit offset in the load itself; 64-bit address arithmetic per lane and row took
// about a quarter of the first pass's instructions and 16 registers.
template <class St, int MAP, bool TWO_D, bool EDGE> struct QuadPull {
    static constexpr bool COL = MAP == kMapCol, SPLIT = MAP == kMapSplit;
    static_assert(!COL || TWO_D, "two rows per lane need ny > 1");
    struct Half {
        float2 C[2], B[2], C2[2], B2[2]; // kMapRow: the neighbour in B.x, B2.x; kMapCol: the pull row in C2.x, B2.x
    };
    static constexpr int ES = int(sizeof(St));
    using Off = std::conditional_t<EDGE, long long, unsigned>; // a lane's byte offset from the tile corner's column
    const char *pa, *pb, *pu, *pd; // at the tile's first column (uniform): rows y, y + 1 (kMapCol), the pull rows of the
                                   // upward and downward populations
    Off oc, om, op, oc2, om2, op2; // the lane's site, its left and right neighbours; the second site's (kMapSplit)
    // base: the populations' first byte in the input buffer, the same for the warp
    __device__ __forceinline__ QuadPull(const KernelArgs &a, const QuadTile<MAP> &t, const char *base)
    {
        constexpr int RIGHT = MAP == kMapRow ? 2 : 1;
        const int yb = COL ? (t.y + 1 < a.ny ? t.y + 1 : bc_index(a.ny, a.ny, a.bcy)) : t.y;
        const int yu = TWO_D ? bc_index(t.y - 1, a.ny, a.bcy) : t.y;
        const int yd = TWO_D ? (COL ? bc_any(t.y + 2, a.ny, a.bcy) : bc_index(t.y + 1, a.ny, a.bcy)) : t.y;
        auto row = [&](int y) { return base + ((long long)y * a.nx + t.x0) * ES; };
        pa = row(t.y);
        pb = row(yb);
        pu = row(yu);
        pd = row(yd);
        auto off = [&](int x) { return Off(x - t.x0) * ES; };
        oc = off(t.x);
        om = off(EDGE ? bc_index(t.x - 1, a.nx, a.bcx) : t.x - 1);
        op = off(EDGE ? bc_index(t.x + RIGHT, a.nx, a.bcx) : t.x + RIGHT);
        oc2 = off(t.x2);
        om2 = SPLIT ? off(EDGE ? bc_index(t.x2 - 1, a.nx, a.bcx) : t.x2 - 1) : 0;
        op2 = SPLIT ? off(EDGE ? bc_index(t.x2 + 1, a.nx, a.bcx) : t.x2 + 1) : 0;
    }
    // off: bytes to population u = 0 of the quad, KS: to its next population
    template <int H> __device__ __forceinline__ void load(Half &b, long long off, long long KS) const
    {
        constexpr int RIGHT = MAP == kMapRow ? 2 : 1;
        // interior: fixed distances from the lane's own offset; a left neighbour is one element
        // before the row's address, so that the 32-bit offset stays positive
        auto centre = [&](const char *row) { return reinterpret_cast<const St *>(row + oc); };
        auto beside = [&](const char *row, bool left) {
            if (EDGE) return reinterpret_cast<const St *>(row + (left ? om : op));
            return reinterpret_cast<const St *>((row + (left ? -ES : RIGHT * ES)) + oc);
        };
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            constexpr bool L0 = H == 0;
            const int u = H + 2 * v;
            const bool left = L0 ? v == 0 : v == 1; // u = 0 and u = 3 pull from x - 1
            const long long o = off + u * KS;
            const char *ra = pa + o;
            if (MAP == kMapRow) {
                b.C[v] = PIo<St>::ld2(centre(ra));
                b.B[v].x = PIo<St>::ld1(beside(ra, left));
                if (TWO_D) {
                    const char *rr = (u < 2 ? pu : pd) + o;
                    b.C2[v] = PIo<St>::ld2(centre(rr));
                    b.B2[v].x = PIo<St>::ld1(beside(rr, left));
                }
            } else if (SPLIT) {
                auto at = [&](Off x) { return PIo<St>::ld1(reinterpret_cast<const St *>(ra + x)); };
                b.C[v] = f2(at(oc), at(oc2));
                b.B[v] = EDGE ? f2(at(left ? om : op), at(left ? om2 : op2))
                              : f2(PIo<St>::ld1(beside(ra, left)), PIo<St>::ld1(beside(ra, left) + 32));
            } else {
                const char *rb = pb + o, *rr = (u < 2 ? pu : pd) + o;
                b.C[v] = f2(PIo<St>::ld1(centre(ra)), PIo<St>::ld1(centre(rb)));
                b.B[v] = f2(PIo<St>::ld1(beside(ra, left)), PIo<St>::ld1(beside(rb, left)));
                b.C2[v].x = PIo<St>::ld1(centre(rr));
                b.B2[v].x = PIo<St>::ld1(beside(rr, left));
            }
        }
    }
    // f[H], f[H + 2] from the loaded half; t0 = (c, c, s, s) of the quad
    template <int H> static __device__ __forceinline__ void pull(const Half &b, float4 t0, float2 *f)
    {
        const float2 c = f2(t0.x, t0.y), s = f2(t0.z, t0.w);
        const float2 ax = H ? s : c, ay = H ? c : s;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const bool left = H == 0 ? v == 0 : v == 1, up = v == 0;
            const float2 cc = b.C[v];
            float2 w;
            if (MAP == kMapRow) {
                w = left ? lerp_x<true>(cc, b.B[v].x, ax) : lerp_x<false>(cc, b.B[v].x, ax);
                if (TWO_D) {
                    const float2 h = left ? lerp_x<true>(b.C2[v], b.B2[v].x, ax) : lerp_x<false>(b.C2[v], b.B2[v].x, ax);
                    w = pfma(ay, psub(h, w), w);
                }
            } else {
                w = pfma(ax, psub(b.B[v], cc), cc);
                if (COL) {
                    const float h = __fmaf_rn(ax.x, b.B2[v].x - b.C2[v].x, b.C2[v].x); // the pull row
                    const float in = up ? w.x - w.y : w.y - w.x;
                    w = pfma(ay, up ? f2(h - w.x, in) : f2(in, h - w.y), w);
                }
            }
            f[H + 2 * v] = w;
        }
    }
};

// The relaxed populations of a quad into the output (Eq. discrete-rbe), rounded
// stochastically.  base: as in QuadPull, in the output buffer.
template <class St, int MAP> struct QuadOut {
    char *pa, *pb;    // rows of the first and second site at the tile's first column (uniform)
    unsigned oa, ob;  // the lane's byte offsets (kMapRow: one paired store)
    bool act0, act1;
    __device__ __forceinline__ QuadOut(const KernelArgs &a, const QuadTile<MAP> &t, char *base)
    {
        constexpr unsigned ES = sizeof(St);
        pa = base + ((long long)t.y * a.nx + t.x0) * ES;
        pb = pa + (MAP == kMapCol && t.y + 1 < a.ny ? (long long)a.nx * ES : 0ll);
        oa = unsigned(t.x - t.x0) * ES;
        ob = unsigned(t.x2 - t.x0) * ES;
        act0 = t.act0;
        act1 = t.act1;
    }
    __device__ __forceinline__ void store(long long off, long long KS, const float2 *f, const float2 *feq,
                                          const float2 *om, QuadBits &rng) const
    {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long o = off + u * KS;
            if constexpr (sizeof(St) == 4) {
                const float2 out = quad_relax_sr(f[u], om[u], feq[u], rng.next());
                if (MAP == kMapRow) {
                    if (act0) *reinterpret_cast<float2 *>(pa + o + oa) = out;
                } else {
                    if (act0) *reinterpret_cast<float *>(pa + o + oa) = out.x;
                    if (act1) *reinterpret_cast<float *>(pb + o + ob) = out.y;
                }
            } else {
                const unsigned d = cvt2_rs<St>(pfma(om[u], psub(feq[u], f[u]), f[u]), rng.next());
                if (MAP == kMapRow) {
                    if (act0) *reinterpret_cast<unsigned *>(pa + o + oa) = d;
                } else {
                    if (act0) *reinterpret_cast<unsigned short *>(pa + o + oa) = (unsigned short)d;
                    if (act1) *reinterpret_cast<unsigned short *>(pb + o + ob) = (unsigned short)(d >> 16);
                }
            }
        }
    }
};

// The step kernel with plain loads: CTA = 64 sites x all populations, warp (q, r) = PP / 4
// quads of shell r, f* of them in registers between the passes.
// QUANT: a quantum statistic (FP32 storage).
template <class St, int N, int PP, int MAP, bool TWO_D, bool QUANT>
__global__ void __maxnreg__(PP <= 16 ? 64 : 128) rlbm_quad_kernel(const KernelArgs a)
{
    constexpr int NC = 2 * N + 1, QW = PP / 4;
    constexpr bool DD = sizeof(St) == 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x, Gs = blockDim.y, K4 = a.K >> 2;
    const int q = warp_uniform(threadIdx.y), r = warp_uniform(threadIdx.z);
    const int g = r * Gs + q, G = Gs * (N + 1);
    const int i0 = r * a.K + q * QW; // population u = 0 of the warp's first quad
    const QuadTile<MAP> t(a, blockIdx.x, blockIdx.y, lane);
    float *red = reinterpret_cast<float *>(smem_raw); // [5][G][64]
    float *sres = red + 5 * G * kPairSites;           // [pair_site_rows(N)][64]
    const float4 *tb = reinterpret_cast<const float4 *>(a.quadtab) + size_t(r * K4 + q * QW) * 3;
    const unsigned seed = __ldcg(a.ctr); // early: its latency passes behind the loads
    // bytes to the next quad's population, to the quad's next (addresses by 64-bit
    // additions: a 64-bit multiply-add takes four cycles of the FMA pipe)
    const long long Sb = a.S * (long long)sizeof(St), KS = K4 * Sb;

    float2 fs[PP];
    QuadSums sums = quad_sums_zero();
    auto pass1 = [&](auto edge_tag) {
        using Pull = QuadPull<St, MAP, TWO_D, decltype(edge_tag)::value>;
        const Pull p(a, t, reinterpret_cast<const char *>(a.fin) + i0 * Sb);
        // the loads run DEPTH - 1 halves ahead of the arithmetic
        constexpr int NH = 2 * QW, DEPTH = PP >= 24 ? 3 : 2;
        typename Pull::Half b[DEPTH];
        auto load = [&](int h) {
            if (h & 1) p.template load<1>(b[h % DEPTH], (h >> 1) * Sb, KS);
            else p.template load<0>(b[h % DEPTH], (h >> 1) * Sb, KS);
        };
#pragma unroll
        for (int h = 0; h < DEPTH - 1; ++h) load(h);
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            if (h + DEPTH - 1 < NH) load(h + DEPTH - 1);
            const int k = h >> 1;
            const float4 t0 = __ldg(tb + 3 * k);
            if (h & 1) {
                Pull::template pull<1>(b[h % DEPTH], t0, fs + 4 * k);
                sums.add(t0, __ldg(tb + 3 * k + 1), fs + 4 * k);
            } else {
                Pull::template pull<0>(b[h % DEPTH], t0, fs + 4 * k);
            }
        }
    };
    if (t.interior(a)) pass1(QuadTag<false>{});
    else pass1(QuadTag<true>{});
    sums.store(reinterpret_cast<float2 *>(red), G, g, lane);
    quad_site<N, DD, QUANT>(a, red, G, Gs, G, g, lane, blockIdx.x + blockIdx.y, sres,
                            [&](int s) { return t.site(a, s); });

    float2 cf[NC], o[3];
    quad_shell<N, DD>(a, r, r, q, Gs, sres, red, lane, cf, o);
    QuadBits rng = quad_seed(unsigned(t.y) * unsigned(a.nx) + unsigned(t.x), unsigned(g), seed);
    const QuadOut<St, MAP> out(a, t, reinterpret_cast<char *>(a.fout) + i0 * Sb);
#pragma unroll
    for (int k = 0; k < QW; ++k) {
        const float4 tq[3] = {__ldg(tb + 3 * k), __ldg(tb + 3 * k + 1),
                              N == 3 ? __ldg(tb + 3 * k + 2) : make_float4(0.f, 0.f, 0.f, 0.f)};
        float2 feq[4], om[4];
        quad_equilibrium<N>(cf, o, tq, feq, om);
        if (k > 0 && 4 * k % QuadBits::kWords == 0) rng.refresh();
        out.store(k * Sb, KS, fs + 4 * k, feq, om, rng);
    }
    __syncthreads();
    if (g == 0 && lane == 0) advance_launch_counter(a.ctr, gridDim.x * gridDim.y);
}

template <class St, int N, int PP, bool QUANT>
static cudaError_t launch_quad_np(int map, bool two_d, dim3 block, size_t smem, cudaStream_t st, const KernelArgs &a)
{
    void (*k)(const KernelArgs) = nullptr;
    dim3 grid((a.nx + 63) / 64, a.ny);
    if (map == kMapCol) {
        k = rlbm_quad_kernel<St, N, PP, kMapCol, true, QUANT>;
        grid = dim3((a.nx + 31) / 32, (a.ny + 1) / 2);
    } else if (map == kMapSplit) {
        k = rlbm_quad_kernel<St, N, PP, kMapSplit, false, QUANT>;
    } else if constexpr (!QUANT) { // the statistics run the forms for any nx only
        if (map == kMapRow)
            k = two_d ? rlbm_quad_kernel<St, N, PP, kMapRow, true, false> : rlbm_quad_kernel<St, N, PP, kMapRow, false, false>;
    }
    if (!k) return cudaErrorInvalidValue;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<grid, block, smem, st>>>(a);
    return cudaGetLastError();
}

// The instances of storage St and order N (one compile unit each).
template <class St, int N, bool QUANT = false>
static cudaError_t launch_quad_n(int PP, int map, bool two_d, dim3 block, size_t smem, cudaStream_t st,
                                 const KernelArgs &a)
{
    switch (PP) {
    case 8: return launch_quad_np<St, N, 8, QUANT>(map, two_d, block, smem, st, a);
    case 12: return launch_quad_np<St, N, 12, QUANT>(map, two_d, block, smem, st, a);
    case 16: return launch_quad_np<St, N, 16, QUANT>(map, two_d, block, smem, st, a);
    case 24: return launch_quad_np<St, N, 24, QUANT>(map, two_d, block, smem, st, a);
    case 32: return launch_quad_np<St, N, 32, QUANT>(map, two_d, block, smem, st, a);
    default: return cudaErrorInvalidValue;
    }
}

} // namespace rlbmk
