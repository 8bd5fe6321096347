"""Free streaming of thin grids with several steps per launch (csrc/rlbm_free.cu) against the
FP64 oracle: 1 to 4 rows, both boundary conditions in x and y, grids smaller than the columns
of a warp, one column around the columns that a warp writes (256 - steps), step counts around
the steps of a launch (32).  FP64: the bound of the other FP64 parity tests.  FP32: every step
rounds once in each of its two interpolations, half a unit (2^-24) of a value that no
interpolation enlarges."""
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


@pytest.mark.parametrize("nx,ny,bcx,bcy", [(1, 1, OUT, PER), (7, 1, PER, PER), (31, 4, PER, OUT), (223, 1, OUT, PER),
                                           (224, 2, PER, PER), (225, 3, OUT, OUT), (1001, 1, PER, PER), (449, 4, OUT, PER)])
@pytest.mark.parametrize("N,K,steps", [(3, 12, 1), (2, 5, 31), (2, 16, 32), (5, 12, 33), (3, 30, 70)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_free_streaming_matches_oracle(nx, ny, bcx, bcy, N, K, steps, precision):
    q = O.Quadrature(N, K)
    f0 = W.random_populations(q.npop, ny, nx, seed=nx + steps) * q.w[:, None, None]
    f0 = f0 if precision == "fp64" else f0.astype(np.float32).astype(np.float64)
    ref, _ = q.run(f0, math.inf, steps, bcx, bcy)
    with R.Simulation(nx, ny, N, K, math.inf, precision, bcx, bcy) as sim:
        sim.set_populations(f0 if precision == "fp64" else f0.astype(np.float32))
        sim.step(steps)
        sim.sync()
        got = sim.get_populations().astype(np.float64)
        assert sim.steps_done == steps
    tol = 1e-12 if precision == "fp64" else 6 * steps * 2.0 ** -24
    scale = np.abs(ref).max(axis=(1, 2), keepdims=True)
    assert np.max(np.abs(got - ref) / scale) < tol
