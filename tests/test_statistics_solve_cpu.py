"""The FP32-storage Fermi-Dirac solve (stat_solve_fd_short and what it declines, rlbm_stat.cuh
compiled into the host library) over its whole range of eta, from cold and warm starts, against
states made from eta itself.

phi_s comes from its definition: the alternating series for eta <= -1, and for eta >= 1 the
inversion identity with that series at -eta (both converge like e^-|eta| per term).

Bounds.  Up to eta = 30 the last FP64 step is below 3e-6 (1 + |eta|), corrected to second order:
what remains is that step times the FP32 rounding of its slope, 3e-6 x 6e-8 = 2e-13, with a
factor ten for the slope's own conditioning.  Beyond, the general solve takes over where the
short one declines: a first-order step below 1e-5 (1 + |eta|), squared, with the same factor
ten: 1e-9; the rounding of n and e, 1e-16 eta^2, stays below that."""
import math

import numpy as np
import pytest

from paper_2011_06856_gb300 import build as B
from paper_2011_06856_gb300 import rlbm as R


def series(s, x):
    return sum((-1) ** (k + 1) * x ** k / k ** s for k in range(1, 60))


def phi(s, eta):
    if eta <= -1.0:
        return series(s, math.exp(eta))
    p2 = math.pi ** 2
    poly = {1: eta, 2: eta ** 2 / 2 + p2 / 6, 3: eta ** 3 / 6 + p2 / 6 * eta}[s]
    return poly + (series(s, math.exp(-eta)) if s & 1 else -series(s, math.exp(-eta)))


@pytest.mark.parametrize("eta", [-50.0, -21.0, -7.5, -1.0, 1.0, 2.7, 6.0, 13.0, 29.0, 40.0, 59.5, 60.5, 100.0, 180.0, 400.0, 650.0])
def test_fp32_storage_fermi_dirac_solve_over_its_range(eta):
    B.build()
    tol = 2e-12 if eta <= 30.0 else 1e-9
    phi2, phi3 = phi(2, eta), phi(3, eta)
    for i in range(400):
        T, g = 0.1 * 1.012 ** i, (0.1, 1.0, 4.0)[i % 3]
        n, e = 2 * math.pi * g * T * T * phi2, 4 * math.pi * g * T ** 3 * phi3
        for d in (math.nan, 0.0, 1e-5 * (i - 200), 1e-3 * (i - 200)):
            got, Tgot, ok = R.quantum_solve(n, e, g, "fd", eta + d * abs(eta), "fp32")
            assert ok
            assert abs(got - eta) < tol * (1 + abs(eta)), (T, g, d, got)
            assert abs(Tgot - T) < 2 * tol * T, (T, g, d, Tgot)


@pytest.mark.parametrize("lo,hi", [(30.0, 60.0), (60.0, 200.0), (200.0, 690.0)])
def test_fp32_storage_fermi_dirac_solve_degenerate(lo, hi):
    """Many states and starts: what the short solve accepts there depends on the FP32 rounding of
    each state."""
    B.build()
    rng = np.random.default_rng(7)
    for eta in rng.uniform(lo, hi, 6000):
        T, g = 10.0 ** rng.uniform(-1, 1), 10.0 ** rng.uniform(-1, 1)
        n, e = 2 * math.pi * g * T * T * phi(2, eta), 4 * math.pi * g * T ** 3 * phi(3, eta)
        got, _, ok = R.quantum_solve(n, e, g, "fd", eta + 1e-3 * (1 + eta) * rng.uniform(-1, 1), "fp32")
        assert ok and abs(got - eta) < 1e-9 * (1 + eta), (eta, T, g, got)
