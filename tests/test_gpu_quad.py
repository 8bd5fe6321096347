"""The quadrant step kernel (csrc/rlbm_quad.cuh) against the FP64 oracle, at the sizes
where its forms can go wrong: every way a lane's two sites lie (one row for an even nx; two
rows for ny > 1 and any nx, with an odd number of rows; 32 apart for ny = 1), grids smaller
than a tile, one cell or one row beyond a tile, both boundary conditions, one, two and four
warps per shell, N = 2 and 3.

FP64 storage (csrc/rlbm_quad64.cuh): the bound of the other FP64 parity tests.  Fermi-Dirac and
Bose-Einstein: the FP32 bound, on rows the statistics' own tests do not have.

FP32 storage: the bound of the other FP32 parity tests (FP32 arithmetic per population, a few
steps).  16-bit storage: stochastic rounding adds at most one unit in the last place per value
and step (2^-10 for FP16, 2^-7 for BF16), which the moments average over the populations; the
bounds are those units."""
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
FP32_TOL = 1e-5
PER, OUT = W.BC_PERIODIC, W.BC_COPYOUT


def relerr(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


def run_both(nx, ny, N, K, tau, precision, bcx, bcy, P, kind, steps):
    fl = W.random_fields(nx, ny, seed=3 * nx + 11 * ny + K)
    q = O.Quadrature(N, K)
    ref, flagged = q.run(q.init(fl.n, fl.T, fl.bx, fl.by), tau, steps, bcx, bcy)
    assert flagged == 0
    with R.Simulation(nx, ny, N, K, tau, precision, bcx, bcy) as sim:
        sim.set_tiling(P, kind)
        assert sim.step_kernel == kind
        sim.init_fields(fl)
        sim.step(steps)
        sim.sync()
        return R.decode_populations(sim.get_populations(), precision, q.w), sim.moments(), ref, q.macro(ref)[0]


@pytest.mark.parametrize("nx,ny,bcx,bcy", [
    (1, 1, PER, PER), (1, 2, OUT, PER), (2, 3, PER, OUT), (31, 2, PER, PER), (33, 5, OUT, OUT), (63, 1, OUT, PER),
    (64, 4, PER, PER), (65, 1, PER, PER), (66, 3, OUT, PER), (97, 7, PER, OUT), (129, 1, OUT, PER), (130, 2, PER, PER)])
@pytest.mark.parametrize("N,K,P", [(2, 8, 8), (2, 24, 12), (3, 32, 8), (3, 16, 16), (2, 48, 24), (3, 64, 32)])
def test_fp32_any_row_length(nx, ny, bcx, bcy, N, K, P):
    for kind in ("per-tile", "pair") if nx % 2 == 0 else ("per-tile",):
        f, _, ref, _ = run_both(nx, ny, N, K, 2.5, "fp32", bcx, bcy, P, kind, 5)
        assert relerr(f, ref) < FP32_TOL, kind


@pytest.mark.parametrize("nx,ny,bcx,bcy", [(1, 1, PER, PER), (31, 2, PER, PER), (33, 5, OUT, OUT), (63, 1, OUT, PER),
                                           (64, 4, PER, PER), (97, 3, PER, OUT)])
@pytest.mark.parametrize("N,K,P", [(2, 8, 8), (2, 24, 12), (3, 32, 8), (3, 16, 16), (2, 48, 24), (3, 64, 32)])
def test_fp64_any_row_length(nx, ny, bcx, bcy, N, K, P):
    f, m, ref, mac = run_both(nx, ny, N, K, 2.5, "fp64", bcx, bcy, P, "per-tile", 5)
    assert relerr(f, ref) < 1e-12 and relerr(m, mac) < 1e-12


@pytest.mark.parametrize("stat", ["fd", "be"])
@pytest.mark.parametrize("N,K,P,nx,ny", [(2, 16, 8, 9, 3), (3, 12, 12, 33, 2), (2, 24, 24, 35, 1)])
def test_fp32_statistics_any_row_length(stat, N, K, P, nx, ny):
    from oracle import statistics as S
    eps, g = {"fd": S.FD, "be": S.BE}[stat], 1.0
    fl = W.random_fields(nx, ny, seed=5, beta_max=0.2)
    fl.n[:] *= 0.5  # fugacities below 1 for the Bose-Einstein runs
    q = O.Quadrature(N, K)
    ref = S.run(q, S.init(q, fl.n, fl.T, fl.bx, fl.by, eps, g), 3.0, 3, OUT, PER, eps, g)
    with R.Simulation(nx, ny, N, K, 3.0, "fp32", OUT, PER) as sim:
        sim.set_statistics(stat, g)
        sim.set_tiling(P, "per-tile")
        sim.init_fields(fl)
        sim.step(3)
        sim.sync()
        assert relerr(sim.get_populations().astype(np.float64), ref) < FP32_TOL


@pytest.mark.parametrize("precision,tol", [("fp16n", 2.0 ** -10), ("fp16", 2.0 ** -10), ("bf16n", 2.0 ** -7), ("bf16", 2.0 ** -7)])
@pytest.mark.parametrize("nx,ny,bcx,bcy", [(33, 5, OUT, OUT), (65, 1, PER, PER), (97, 2, PER, OUT), (96, 3, OUT, PER)])
def test_16bit_any_row_length(nx, ny, bcx, bcy, precision, tol):
    steps = 2
    f, m, ref, mac = run_both(nx, ny, 2, 48, 3.0, precision, bcx, bcy, 24, "per-tile", steps)
    w = O.Quadrature(2, 48).w[:, None, None] / (2.0 * np.pi)
    stored = np.abs(ref / w).max() + 1.0
    assert np.max(np.abs(f - ref) / w) < (steps + 1) * tol * stored
    assert relerr(m[:2], mac[:2]) < steps * tol


def test_unphysical_cell_is_reported_only_inside_the_grid():
    """Ragged tiles and a missing second row solve copies of grid cells: no false report; a
    cell without a physical frame is reported."""
    nx, ny, N, K = 33, 3, 2, 24
    q = O.Quadrature(N, K)
    fl = W.random_fields(nx, ny, seed=8)
    with R.Simulation(nx, ny, N, K, 3.0, "fp32", OUT, OUT) as sim:
        sim.set_tiling(12, "per-tile")
        sim.init_fields(fl)
        sim.step(3)
        sim.sync()
        f = q.init(fl.n, fl.T, fl.bx, fl.by).astype(np.float32)
        f[:, ny - 1, nx - 1] *= -1.0
        sim.set_populations(f)
        sim.step(1)
        with pytest.raises(R.Unphysical):
            sim.sync()


# Many angles: two passes in one launch (csrc/rlbm_quad_split.cuh).  K / 4 even and odd, fewer
# quads per CTA than warps, more; each way a lane's two sites lie; P is a tiling that leaves K
# to the two passes; the widest grid has more tiles than the ring has places.
@pytest.mark.parametrize("nx,ny,bcx,bcy", [(1, 1, PER, PER), (33, 3, OUT, OUT), (63, 1, OUT, PER), (66, 2, PER, OUT),
                                           (130, 1, PER, PER)])
@pytest.mark.parametrize("N,K,P", [(2, 100, 64), (3, 120, 48), (3, 120, 64), (2, 300, 64), (3, 288, 12), (2, 600, 24)])
def test_fp32_many_angles(nx, ny, bcx, bcy, N, K, P):
    pair = nx % 2 == 0 and K % P == 0 and P <= 32
    for kind in ("per-tile", "pair") if pair else ("per-tile",):
        f, m, ref, mac = run_both(nx, ny, N, K, 2.5, "fp32", bcx, bcy, P, kind, 4)
        assert relerr(f, ref) < FP32_TOL and relerr(m[:2], mac[:2]) < FP32_TOL, kind


@pytest.mark.parametrize("precision", ["fp32", "fp16n"])
def test_many_angles_more_tiles_than_ring_places(precision):
    nx, ny, N, K = 513, 192, 2, 68
    fl = W.random_fields(nx, ny, seed=4)
    mom = {}
    for p in (precision, "fp64"):
        with R.Simulation(nx, ny, N, K, 2.5, p, OUT, PER) as sim:
            sim.set_tiling(48, "per-tile")
            sim.init_fields(fl)
            sim.step(2)
            sim.sync()
            mom[p] = sim.moments()
    assert relerr(mom[precision][:2], mom["fp64"][:2]) < (FP32_TOL if precision == "fp32" else 2 * 2.0 ** -10)


def test_many_angles_report_an_unphysical_cell():
    nx, ny, N, K = 33, 3, 3, 288
    q = O.Quadrature(N, K)
    fl = W.random_fields(nx, ny, seed=8)
    with R.Simulation(nx, ny, N, K, 3.0, "fp32", OUT, OUT) as sim:
        sim.init_fields(fl)
        sim.step(2)
        sim.sync()
        f = q.init(fl.n, fl.T, fl.bx, fl.by).astype(np.float32)
        f[:, ny - 1, nx - 1] *= -1.0
        sim.set_populations(f)
        sim.step(1)
        with pytest.raises(R.Unphysical):
            sim.sync()


def test_many_angles_expired_wait_is_reported_and_recovered_from():
    """With a wait limit far below a tile's first pass the second pass gives up: the step is
    reported, and the same handle steps correctly afterwards (its counters start over)."""
    nx, ny, N, K = 96, 4, 3, 288
    fl = W.random_fields(nx, ny, seed=9)
    q = O.Quadrature(N, K)
    ref, flagged = q.run(q.init(fl.n, fl.T, fl.bx, fl.by), 2.5, 3, OUT, PER)
    assert flagged == 0
    with R.Simulation(nx, ny, N, K, 2.5, "fp32", OUT, PER) as sim:
        sim.init_fields(fl)
        sim.set_wait_limit(1000)
        sim.step(1)
        with pytest.raises(R.DeviceTimeout):
            sim.sync()
        sim.set_wait_limit(4_000_000_000)
        sim.init_fields(fl)
        sim.step(3)
        sim.sync()
        assert relerr(sim.get_populations().astype(np.float64), ref) < FP32_TOL
