"""The closure's tensor-core kernels at the edges of their tiles: one site, one less and one
more than the 16 rows of a warp, than the 128 columns of a training tile; every specialised
rule.

The references carry the same BF16 roundings; what is left are values whose FP32 and FP64
sums lie on either side of a rounding boundary: one BF16 unit (2^-8 relative) of one factor
of a product, two where both factors of a weight gradient flip.  With few columns nothing
averages that, so the bounds are those units of the largest value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2011_06856_gb300 import rlbm as R  # noqa: E402
from test_gpu_closure import apply_case, bf16_loss_and_grad, ref_params  # noqa: E402

RULES = [(2, 24), (2, 16), (3, 16)]


@pytest.mark.parametrize("n,k", RULES)
@pytest.mark.parametrize("count", [1, 15, 17, 127, 129])
def test_gradient_at_tile_edges(n, k, count):
    cl = R.Closure(n, k, seed=5)
    g = np.random.default_rng(100 * n + k + count)
    S, off = count + 7, 3
    X = g.normal(0, 0.5, (cl.F, S)).astype(np.float32)
    T = g.normal(0, 0.1, (cl.npop, S)).astype(np.float32)
    grad, loss = cl.gradient(torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda"), off, count, cl.work(S))
    lb, gb = bf16_loss_and_grad(ref_params(cl), X[:, off:off + count].T.astype(np.float64),
                                T[:, off:off + count].T.astype(np.float64))
    flat = np.concatenate([a.ravel() for a in gb])
    assert abs(loss - lb) < 2.0 ** -8 * lb
    assert np.abs(grad - flat).max() < 2.0 ** -7 * np.abs(flat).max()


@pytest.mark.parametrize("n,k", RULES)
@pytest.mark.parametrize("sites", [1, 15, 17, 255, 257])
def test_apply_at_group_edges(n, k, sites):
    q, f32, got, ref, d, Cm = apply_case(sites, 40 + sites, True, n, k)
    np.testing.assert_allclose(got, ref, rtol=1e-4, atol=2.0 ** -7 * np.abs(d).max())
    before, after = Cm @ f32, Cm @ got
    assert np.abs(after - before).max() < 2e-6 * np.abs(before).max()
