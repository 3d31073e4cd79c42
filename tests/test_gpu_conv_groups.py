"""The learned correction's convolutions in groups of eight sites per thread (116736 (site, column) pairs and
more) with the block width known at compile time (16, 32, 64) and at run time, and in groups of
four below, on sides that the groups do not divide (the last group of a row is moved back):
inference, the tap-by-tap forward pass and the masked data gradients of the loss gradient, periodic
complex and Dirichlet real (zero halos).  Bounds: forward 1e-5, loss 1e-4, gradient 1e-3 of scale."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import learned as NN
from oracle.operators import laplace2d, wilson2d
from paper_2108_11281_gb300.workloads import gauge_links


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


@pytest.mark.parametrize("op", ["wilson", "laplace"])
@pytest.mark.parametrize("nx,ny,k", [(92, 92, 16), (68, 60, 32), (44, 44, 64), (52, 48, 48), (44, 44, 40), (4, 1828, 16)])
def test_network_and_gradient_match_oracle(mlmc, op, nx, ny, k):
    kw = dict(levels=2, precision=mlmc.PREC_MIXED_FP32, block=k, bootstrap=0)
    if op == "wilson":
        U = gauge_links(nx, ny, 0.3, 2)
        prm = mlmc.default_params(n_tv=2, spin_split=1, setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=4, setup_omega=1.0, **kw)
        h = mlmc.Hierarchy(mlmc.OP_WILSON2D, nx, ny, prm, mass=0.2, links=U)
        A, d, cplx = wilson2d(nx, ny, 0.2, U), 2, True
    else:
        prm = mlmc.default_params(n_tv=1, setup_kind=mlmc.SETUP_CONSTANT, **kw)
        h, A, d, cplx = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, nx, ny, prm), laplace2d(nx, ny), 1, False
    h.set_conv_kernel(mlmc.CONV_SIMT)
    Ws = [W.astype(np.float32).astype(np.float64) for W in NN.init_weights(NN.channels_of(d, cplx), 9)]
    h.learned_set(np.concatenate([W.astype(np.float32).ravel() for W in Ws]), enable=0)
    R = torch.randn(nx * ny * d, k, dtype=torch.complex64 if cplx else torch.float32, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(nx + k))
    E = torch.full_like(R, float("nan"))
    h.learned_apply(R.data_ptr(), E.data_ptr(), k)
    loss, grad = h.learned_grad(R.data_ptr(), k)
    h.close()
    Rn, En = R.cpu().numpy().astype(np.complex128 if cplx else np.float64), E.cpu().numpy()
    assert np.isfinite(En).all()
    for c in range(0, k, 5):
        ref, _ = NN.forward(Rn[:, c], Ws, nx, ny, d, cplx, cplx)
        assert np.abs(En[:, c] - ref).max() <= 1e-5 * np.abs(ref).max()
    ref_loss, ref_g = NN.loss_and_grad(A, Rn, Ws, nx, ny, d, cplx, cplx)
    ref_flat = np.concatenate([x.ravel() for x in ref_g])
    assert abs(loss - ref_loss) <= 1e-4 * abs(ref_loss)
    assert np.abs(grad - ref_flat).max() <= 1e-3 * np.abs(ref_flat).max()
