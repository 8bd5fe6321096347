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
