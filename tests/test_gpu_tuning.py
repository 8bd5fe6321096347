"""The autotuner's process-wide cache (rlbm_autotune)."""
import math

import pytest

from paper_2011_06856_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2011_06856_gb300 import build as B  # noqa: E402
from paper_2011_06856_gb300 import rlbm as R  # noqa: E402

B.build()


def test_free_streaming_and_collisions_are_tuned_apart():
    """A free-streaming handle can run two of the step kernels only, and its steps do no
    collision: its choice is not the one for a handle of the same shape with a finite tau.  Two
    handles that share an entry report the same time to the bit; a collision step in FP64 takes
    several times as long as a streaming step (38 against 9 FP64 operations per population)."""
    nx, ny, N, K = 768, 160, 3, 24
    ms = {}
    for tau in (math.inf, 2.0, math.inf, 2.5):
        with R.Simulation(nx, ny, N, K, tau, "fp64", W.BC_PERIODIC, W.BC_PERIODIC) as sim:
            sim.init_fields(W.uniform(nx, ny, 1.0, 1.0))
            ms.setdefault(math.isinf(tau), []).append(sim.autotune(4))
            again = sim.autotune(4)
            assert again == ms[math.isinf(tau)][-1]
    assert ms[True][0] == ms[True][1] and ms[False][0] == ms[False][1]
    assert ms[False][0] > 1.2 * ms[True][0]
