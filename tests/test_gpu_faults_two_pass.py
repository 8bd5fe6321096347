"""The timeout test hook (rlbm_test_stall_next_step) on the two-pass kernel of many angles: its
second pass waits for more CTAs than a tile has, the bounded wait runs out, the host reads
RLBM_ERR_TIMEOUT and the handle steps correctly afterwards."""
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


@pytest.mark.parametrize("N,K,P,kind", [(2, 288, 64, "per-tile"), (2, 600, 24, "pair")])
def test_stalled_two_pass_step_reports_timeout_and_recovers(N, K, P, kind):
    nx, ny, tau = 96, 4, 2.5
    fl = W.random_fields(nx, ny, seed=2)
    q = O.Quadrature(N, K)
    f0 = q.init(fl.n, fl.T, fl.bx, fl.by)
    with R.Simulation(nx, ny, N, K, tau, "fp32", W.BC_COPYOUT, W.BC_PERIODIC) as sim:
        sim.set_tiling(P, kind)
        sim.init_fields(fl)
        sim.set_wait_limit(2_000_000)  # about 1 ms
        sim.test_stall_next_step()
        sim.step(1)
        with pytest.raises(R.DeviceTimeout):
            sim.sync()
        sim.set_wait_limit(4_000_000_000)
        sim.set_populations(f0.astype(np.float32))
        sim.step(3)
        sim.sync()
        ref, flagged = q.run(f0, tau, 3, W.BC_COPYOUT, W.BC_PERIODIC)
        assert flagged == 0
        got = sim.get_populations().astype(np.float64)
        assert np.abs(got - ref).max() / np.abs(ref).max() < 1e-5
