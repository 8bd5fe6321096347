// Random bits of the quadrant kernels' stochastic rounding; also compiled on the host.
#pragma once

#ifdef __CUDACC__
#define RLBM_BITS __host__ __device__ __forceinline__
#else
#define RLBM_BITS inline
#endif

namespace rlbmk {

RLBM_BITS unsigned mix32(unsigned x)
{
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}

RLBM_BITS unsigned rotl32(unsigned x, int n)
{
#ifdef __CUDA_ARCH__
    return __funnelshift_l(x, x, n);
#else
    return x << n | x >> (32 - n);
#endif
}

// The k-th word of a thread is the exclusive or of two hashed words rotated by 5 k and 3 k
// bits.  Bit i of word k joins bits i - 5 k and i - 3 k of the two, whose distance 2 k comes
// back after 16 words: up to there no pair of bits meets twice, so that any two bits of the
// words are independent, which is what the moments of the rounding errors need; word k + 16
// would be word k with its halves (the lane's two sites) exchanged.  After kWords words the
// first of the two is therefore hashed again (refresh), 8 integer operations per 16 words.
// A word costs three integer operations on the pipe that the arithmetic leaves idle; an LCG
// draw (IMAD) takes two cycles of the FMA pipe, a 64-bit product four.
struct QuadBits {
    static constexpr int kWords = 16;
    unsigned a, b;
    RLBM_BITS unsigned next()
    {
        a = rotl32(a, 5);
        b = rotl32(b, 3);
        return a ^ b;
    }
    RLBM_BITS void refresh() { a = mix32(a + 0x9E3779B9u); }
};

// Seeded by the thread's first site, the warp g < 256 and the launch counter.  The site is
// hashed before the counter enters: the exclusive or of the counter's hash with the bare site
// index only permutes the seeds of a launch among the sites, so that every launch rounds with
// almost the same set of words, and the mean error of that set becomes a drift of n (5e-4
// over 2000 steps of a 256^2 grid in FP16).  Sites 2^24 apart share the first word and differ
// in the second: no two threads of a launch have the same pair.
RLBM_BITS QuadBits quad_seed(unsigned site, unsigned g, unsigned launch)
{
    const unsigned h = mix32(mix32(site * 256u + g) ^ mix32(launch * 0x9E3779B9u + 1u));
    return {h, mix32(h + 0x9E3779B9u + (site >> 24))};
}

} // namespace rlbmk
