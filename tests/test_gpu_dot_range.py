"""Column sums of FP32 data beyond FP32's range: |r|^2 of a column of 1024 entries of 2^60 is 1e39, while a
product and a thread's own sum stay below 3.4e38.  The network has no biases and its ReLUs are
positively homogeneous, so the loss |r - A net(r)|^2 / |r|^2 and its gradient do not change when r
is multiplied by a power of two (nor does any rounding): 1e-6 and 1e-5 of scale."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import learned as NN


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


@pytest.mark.parametrize("k", [1, 2, 4, 33])
def test_loss_of_large_residuals(mlmc, k):
    prm = mlmc.default_params(n_tv=1, setup_kind=mlmc.SETUP_CONSTANT, precision=mlmc.PREC_MIXED_FP32, block=k, bootstrap=0)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, 32, 32, prm)
    W1, W2, W3 = NN.init_weights(1, 9)
    # a small last layer: the residual after the network has r's own size, so its products are in range too
    h.learned_set(np.concatenate([W.astype(np.float32).ravel() for W in (W1, W2, 1e-2 * W3)]), enable=0)
    r = torch.randn(1024, k, dtype=torch.float32, device="cuda", generator=torch.Generator(device="cuda").manual_seed(k))
    loss, grad = h.learned_grad(r.data_ptr(), k)
    big = r * 2.0 ** 60
    loss_big, grad_big = h.learned_grad(big.data_ptr(), k)
    h.close()
    assert (big.double().norm(dim=0) ** 2 > 3.5e38).all() and 0.5 < loss < 2.0
    assert abs(loss_big - loss) <= 1e-6 * loss
    assert np.abs(grad_big - grad).max() <= 1e-5 * np.abs(grad).max()
