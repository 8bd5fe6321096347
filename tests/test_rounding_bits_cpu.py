"""Random bits of the quadrant kernels' stochastic rounding (csrc/rlbm_bits.cuh), compiled for
the host: the words of a thread in the order in which the kernels draw them (hashed again after
every QuadBits::kWords of them), up to 608 draws (2400 angles of a shell by one CTA of four
warps), and the seeds of a launch.

Two words of independent bits differ in 16 +- sqrt(8) of their 32 bits.  Over 4096 threads the
mean is within sqrt(8 / 4096) = 0.044 of 16 (one sigma); 7 sigma are allowed for every pair
of the first 48 words and every rotation of one against the other, 7e4 means."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2011_06856_gb300", "csrc")

PROGRAM = r"""
#include "rlbm_bits.cuh"
using namespace rlbmk;
extern "C" void words(unsigned site, unsigned g, unsigned launch, int n, unsigned *out)
{
    QuadBits r = quad_seed(site, g, launch);
    for (int k = 0; k < n; ++k) {
        if (k > 0 && k % QuadBits::kWords == 0) r.refresh();
        out[k] = r.next();
    }
}
extern "C" void mean_distance(const unsigned *w, int threads, int n, double *out)
{
    for (int j = 0; j < n; ++j)
        for (int k = 0; k < n; ++k)
            for (int s = 0; s < 32; ++s) {
                long long c = 0;
                for (int t = 0; t < threads; ++t) {
                    const unsigned v = w[t * n + k];
                    c += __builtin_popcount(w[t * n + j] ^ (s ? v << s | v >> (32 - s) : v));
                }
                out[(j * n + k) * 32 + s] = double(c) / threads;
            }
}
"""


@pytest.fixture(scope="module")
def bits(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("needs a C++ compiler")
    d = tmp_path_factory.mktemp("bits")
    src, so = d / "bits.cpp", d / "bits.so"
    src.write_text(PROGRAM)
    res = subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return ctypes.CDLL(str(so))


def draw(bits, sites, g, launch, n):
    w = np.zeros((len(sites), n), dtype=np.uint32)
    for t, s in enumerate(sites):
        bits.words(ctypes.c_uint(int(s)), g, launch, n, ctypes.c_void_p(w[t].ctypes.data))
    return w


def rot(w, s):
    return (w << np.uint32(s) | w >> np.uint32(32 - s)).astype(np.uint32) if s else w


@pytest.mark.parametrize("launch", [0, 7])
def test_words_of_a_thread_do_not_repeat(bits, launch):
    """Neither a word nor the word with its halves (the two sites of a lane) exchanged."""
    n = 608
    w = draw(bits, range(0, 128, 2), 3, launch, n)
    for row in w:
        both = np.concatenate([row, rot(row, 16)])
        assert len(np.unique(both)) > 2 * n - 3  # 2^21 pairs of 2^32 values: a chance pair now and then


def test_words_of_a_thread_are_uncorrelated(bits):
    threads, n = 4096, 48
    w = draw(bits, range(threads), 5, 3, n)
    d = np.zeros((n, n, 32))
    bits.mean_distance(ctypes.c_void_p(np.ascontiguousarray(w).ctypes.data), threads, n, ctypes.c_void_p(d.ctypes.data))
    off = ~np.eye(n, dtype=bool)
    assert np.abs(d[off] - 16.0).max() < 7 * np.sqrt(8.0 / threads)


@pytest.mark.parametrize("stride", [1, 2, 64, 1 << 16, 1 << 24, 3 << 24, 1 << 28])
def test_seeds_of_a_launch_are_distinct(bits, stride):
    """The same warp at two sites, and neighbouring warps: other words, of which the first 16
    differ in half their bits on average (sigma sqrt(8 / (16 threads)))."""
    threads = 4096
    base = np.arange(threads, dtype=np.int64) * 5
    a = draw(bits, base, 2, 11, 16)
    for other in (draw(bits, base + stride, 2, 11, 16), draw(bits, base, 3, 11, 16)):
        x = (a ^ other).view(np.uint8)
        mean = np.unpackbits(x).sum() / (threads * 16)
        assert abs(mean - 16.0) < 7 * np.sqrt(8.0 / threads / 16) * 4  # words of a thread share their hash
        assert (a != other).any(axis=1).all()
