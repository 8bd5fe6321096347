"""The stochastic rounding of the quadrant kernels (csrc/rlbm_quad.cuh, rlbm_quad_split.cuh,
rlbm_pair_tma.cuh): the errors of a site's populations are independent of each other and of the
other site of the lane.

One step of a uniform state away from equilibrium: streaming leaves it as it is and every site
computes the same values, so that the sites differ by the rounding noise alone.  With
independent noise the variance over the sites of the first moment sum p_i f_i is the sum of the
populations' own, sum p_i^2 var f_i, and the moments of a lane's two sites are uncorrelated.
Both are known from S sites to sqrt(2 / S) and, over S / 2 pairs, sqrt(2 / S); seven of those
are allowed.  Populations that share their noise (more draws per thread than the generator has
words) would double the variance or correlate the pair by a fifth and more."""
import numpy as np
import pytest

import oracle as O
from paper_2011_06856_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2011_06856_gb300 import build as B  # noqa: E402
from paper_2011_06856_gb300 import rlbm as R  # noqa: E402

B.build()


@pytest.mark.parametrize("precision,N,K,P,kind,nx", [
    ("fp32", 2, 288, 64, "per-tile", 256), ("fp32", 2, 600, 24, "pair", 256), ("fp16n", 2, 288, 64, "per-tile", 255),
    ("fp32", 2, 96, 32, "pair", 256), ("fp32", 2, 96, 32, "per-tile", 255), ("fp32", 2, 48, 24, "per-tile", 256),
    ("fp16n", 2, 96, 32, "pair-tma", 256), ("bf16n", 2, 48, 24, "pair-tma", 256), ("fp16", 3, 24, 12, "pair", 256),
    ("fp32", 3, 64, 16, "per-tile", 255)])
def test_rounding_noise_is_independent(precision, N, K, P, kind, nx):
    ny = 192
    q = O.Quadrature(N, K)
    one = np.ones((1, 1))
    f = q.init(0.9 * one, 1.1 * one, 0.2 * one, -0.1 * one)[:, 0, 0]
    f *= 1.0 + 0.1 * (2.0 * np.random.default_rng(K).random(q.npop) - 1.0)
    s = f / (q.w / (2.0 * np.pi)) - (0.0 if precision.endswith("n") else 1.0)
    if precision == "fp32":
        raw = f.astype(np.float32)
    elif precision.startswith("fp16"):
        raw = s.astype(np.float16)
    else:
        raw = (s.astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)
    with R.Simulation(nx, ny, N, K, 3.0, precision, W.BC_PERIODIC, W.BC_PERIODIC) as sim:
        sim.set_tiling(P, kind)
        sim.set_populations(np.broadcast_to(raw[:, None, None], (q.npop, ny, nx)))
        sim.step(1)
        sim.sync()
        out = R.decode_populations(sim.get_populations(), precision, q.w).reshape(q.npop, -1)
    out -= out.mean(axis=1, keepdims=True)
    m = q.p0 @ out
    tol = 7.0 * np.sqrt(2.0 / m.size)
    assert abs(m.var() / (q.p0 ** 2 @ out.var(axis=1)) - 1.0) < tol
    m = m.reshape(ny, nx)
    for a, b in ((m[:, 0:nx - 1:2], m[:, 1:nx:2]), (m[0::2], m[1::2])):
        assert abs((a * b).mean() / m.var()) < tol


@pytest.mark.parametrize("N,K,P,kind,nx", [(2, 96, 24, "pair", 128), (2, 64, 16, "per-tile", 255), (2, 288, 64, "per-tile", 128),
                                           (2, 48, 16, "pair-tma", 128)])
def test_fp32_store_keeps_the_residual_of_a_strong_relaxation(N, K, P, kind, nx):
    """A uniform state far from equilibrium: every site of a population rounds the same value, to
    one of two neighbours, the upper one with a probability p that is the value's place between
    them, whichever of the two is the even one.  Were the change om (f^eq - f*) rounded to its own
    unit first, an eighth of the result's or more for a change of an eighth of its power of two or
    more, the last rounding would meet ties, and ties go to the even neighbour: p would be larger
    by a sixteenth or more where the upper one is even and smaller where it is odd.  The places are
    uniform in [0, 1] (standard deviation 1 / sqrt(12)), so the means of p over n_e and n_o
    populations differ by 0 +- sqrt((1 / n_e + 1 / n_o) / 12); 5.5 of those are allowed, less than
    the eighth that would show."""
    ny = 200
    q = O.Quadrature(N, K)
    one = np.ones((1, 1))
    p, even = [], []
    with R.Simulation(nx, ny, N, K, 1.6, "fp32", W.BC_PERIODIC, W.BC_PERIODIC) as sim:
        sim.set_tiling(P, kind)
        seed = 0
        while sum(map(len, p)) < 3000:
            f = q.init(0.9 * one, 1.1 * one, 0.2 * one, -0.1 * one)[:, 0, 0]
            f *= 1.0 + 0.5 * (2.0 * np.random.default_rng(seed).random(q.npop) - 1.0)
            raw = f.astype(np.float32)
            sim.set_populations(np.broadcast_to(raw[:, None, None], (q.npop, ny, nx)), step=seed)
            sim.step(1)
            sim.sync()
            out = sim.get_populations().reshape(q.npop, -1)
            lo, hi = out.min(axis=1), out.max(axis=1)
            two_e = 2.0 ** np.floor(np.log2(lo.astype(np.float64)))
            change = np.abs(0.5 * (lo.astype(np.float64) + hi) - raw)
            use = (change > two_e / 8) & (change < 0.5 * raw) & (hi == np.nextafter(lo, np.float32(np.inf))) & (hi < 2 * two_e)
            p.append((out[use] != lo[use, None]).mean(axis=1))
            even.append(hi[use].view(np.uint32) % 2 == 0)
            seed += 1
            assert seed < 200
    p, even = np.concatenate(p), np.concatenate(even)
    bound = 5.5 * np.sqrt((1.0 / even.sum() + 1.0 / (~even).sum()) / 12.0)
    assert bound < 0.1 and abs(p[even].mean() - p[~even].mean()) < bound
