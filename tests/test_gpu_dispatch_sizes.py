"""Both sides of the grid sizes at which kind 0 changes its kernel, against the FP64 oracle: one
or two rows per lane in FP64 (as many tiles of two rows as the GPU has SMs), the quadrant kernel
with P = 16 or the per-tile kernel (two tiles for three SMs in FP32, seven warps per SM in 16-bit
storage), two passes or one group of populations per warp (6144 sites for a ragged tiling, 16384
for a full one).  Odd rows, odd numbers of rows, and the autotuner's choices.  The bounds are
those of the other parity tests of these storage forms."""
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
TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp16n": 2 * 2.0 ** -10}


def run(nx, ny, N, K, precision, tiling):
    fl = W.random_fields(nx, ny, seed=nx + ny + K)
    q = O.Quadrature(N, K)
    ref, flagged = q.run(q.init(fl.n, fl.T, fl.bx, fl.by), 2.5, 2, W.BC_COPYOUT, W.BC_PERIODIC)
    assert flagged == 0
    mac = q.macro(ref)[0][:2]
    with R.Simulation(nx, ny, N, K, 2.5, precision, W.BC_COPYOUT, W.BC_PERIODIC) as sim:
        sim.init_fields(fl)
        if tiling:
            sim.set_tiling(*tiling)
        else:
            sim.autotune(2)
        sim.init_fields(fl)
        sim.step(2)
        sim.sync()
        m = sim.moments()[:2]
        assert np.max(np.abs(m - mac)) / np.max(np.abs(mac)) < TOL[precision]
        if precision != "fp16n":
            f = sim.get_populations().astype(np.float64)
            assert np.max(np.abs(f - ref)) / np.max(np.abs(ref)) < TOL[precision]


@pytest.mark.parametrize("nx,ny", [(33, 149), (33, 305), (64, 152), (1, 303)])
@pytest.mark.parametrize("N,K,P", [(2, 8, 8), (3, 24, 12), (2, 48, 16)])
def test_fp64_rows_per_lane(nx, ny, N, K, P):
    run(nx, ny, N, K, "fp64", (P, "per-tile"))


@pytest.mark.parametrize("nx,ny,precision", [(33, 99, "fp32"), (33, 103, "fp32"), (6463, 1, "fp32"), (6529, 1, "fp32"),
                                             (65, 231, "fp16n"), (65, 237, "fp16n")])
def test_sixteen_populations_per_warp(nx, ny, precision):
    run(nx, ny, 2, 16, precision, (16, "per-tile"))


@pytest.mark.parametrize("nx,ny,K,P,precision", [(65, 93, 68, 24, "fp32"), (65, 95, 68, 24, "fp32"), (6143, 1, 100, 32, "fp32"),
                                                 (127, 128, 128, 64, "fp32"), (127, 130, 128, 64, "fp32"),
                                                 (127, 193, 128, 64, "fp16n"), (127, 195, 128, 64, "fp16n")])
def test_two_passes_or_one(nx, ny, K, P, precision):
    run(nx, ny, 2, K, precision, (P, "per-tile"))


@pytest.mark.parametrize("nx,ny,N,K,precision", [(33, 33, 2, 60, "fp64"), (64, 64, 3, 16, "fp32"), (65, 33, 2, 68, "fp32"),
                                                 (66, 40, 3, 288, "fp32"), (33, 33, 2, 16, "fp16n"),
                                                (8192, 1, 2, 600, "fp32"), (128, 128, 2, 400, "fp32")])
def test_tuned_choice(nx, ny, N, K, precision):
    run(nx, ny, N, K, precision, None)
