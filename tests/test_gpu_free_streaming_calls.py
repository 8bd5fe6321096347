"""Free streaming of thin grids (csrc/rlbm_free.cu) through calls that its launch geometry and
its several steps per launch could change: more populations than a grid dimension holds, and
steps captured into a caller's graph."""
import math

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
PER, OUT = W.BC_PERIODIC, W.BC_COPYOUT


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("K", [16383, 16384, 32800])
def test_more_populations_than_a_grid_dimension(K, precision):
    """(N + 1) K around 65535 and beyond twice that, on a line: the interpolation of Eq.
    interpolation with the columns' upwind neighbours, copied out at both ends.  FP32: two
    roundings of half a unit per step, no value grows."""
    N, nx, steps = 3, 9, 3
    vx = O.Quadrature(N, K).vx[:, None]
    dt = np.float64 if precision == "fp64" else np.float32
    f0 = np.random.default_rng(K).random((vx.size, nx)).astype(dt)
    ref = f0.astype(np.float64)
    for _ in range(steps):
        left = np.concatenate([ref[:, :1], ref[:, :-1]], axis=1)
        right = np.concatenate([ref[:, 1:], ref[:, -1:]], axis=1)
        ref = ref + np.abs(vx) * (np.where(vx >= 0, left, right) - ref)
    with R.Simulation(nx, 1, N, K, math.inf, precision, OUT, PER) as sim:
        sim.set_populations(f0[:, None, :])
        sim.step(steps)
        sim.sync()
        got = sim.get_populations()[:, 0, :].astype(np.float64)
    assert np.max(np.abs(got - ref)) < (1e-12 if precision == "fp64" else 6 * steps * 2.0 ** -24)


@pytest.mark.parametrize("nsteps", [2, 6, 30, 32, 64, 96])
def test_captured_steps_go_on_at_every_replay(nsteps):
    """An even number of steps captured on the handle's stream ends in the buffer it started
    from: each replay advances the state by nsteps, bit for bit as plain steps do."""
    nx, ny, N, K, replays = 300, 2, 2, 12, 3
    f0 = W.random_populations(K * (N + 1), ny, nx, seed=nsteps).astype(np.float32)
    with R.Simulation(nx, ny, N, K, math.inf, "fp32", PER, OUT) as ref:
        ref.set_populations(f0)
        ref.step(replays * nsteps)
        want = ref.get_populations()
    with R.Simulation(nx, ny, N, K, math.inf, "fp32", PER, OUT) as sim:
        sim.set_populations(f0)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=sim.stream):
            sim.step(nsteps)
        for _ in range(replays):
            graph.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(sim.get_populations(), want)
