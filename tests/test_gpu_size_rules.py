"""Sizes at which a kernel's split changes: the FP64 Example 5.1 product on either side of the line
between sites and strips (odd and narrow lattices, odd block widths, walks that end inside the
lattice), and the network with four and with eight sites per thread (also on a lattice narrower than
a group).  At most five products per entry: 1e-13 of the largest; network and gradient as in
test_gpu_learned.py: forward 1e-5, loss 1e-4, gradient 1e-3 of scale."""
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


@pytest.mark.parametrize("nx,ny,periodic,k", [(63, 47, 0, 236), (63, 47, 0, 237), (129, 43, 0, 129), (255, 259, 0, 11),
                                              (256, 128, 1, 21), (256, 128, 1, 22), (12, 232, 1, 256), (4, 684, 1, 256),
                                              (511, 1023, 0, 2), (1024, 1024, 0, 1)])
def test_fp64_laplace(mlmc, nx, ny, periodic, k):
    kw = dict(levels=2 if nx * ny <= 32768 else 4, n_tv=1, block=4, bootstrap=0)
    if nx % 2:
        prm = mlmc.default_params(transfer=mlmc.TRANSFER_BILINEAR, **dict(kw, levels=3 if nx == 255 else kw["levels"]))
    else:
        prm = mlmc.default_params(setup_kind=mlmc.SETUP_CONSTANT, agg_x=4, agg_y=4, **kw)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, nx, ny, prm, shift=0.3, periodic=periodic)
    x = torch.randn(nx * ny, k, dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(nx + k))
    y = torch.full_like(x, float("nan"))
    h.apply(1, x.data_ptr(), y.data_ptr(), k)
    h.close()
    ref = laplace2d(nx, ny, 0.3, bool(periodic)) @ x.cpu().numpy()
    assert np.abs(y.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("nx,ny,k", [(36, 36, 64), (20, 60, 61), (40, 40, 80), (52, 52, 48), (36, 60, 55), (4, 256, 128)])
def test_network_and_gradient(mlmc, nx, ny, k):
    U = gauge_links(nx, ny, 0.3, 2)
    prm = mlmc.default_params(levels=2, n_tv=2, spin_split=1, setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=4,
                              setup_omega=1.0, precision=mlmc.PREC_MIXED_FP32, block=k, bootstrap=0)
    h = mlmc.Hierarchy(mlmc.OP_WILSON2D, nx, ny, prm, mass=0.2, links=U)
    A, d = wilson2d(nx, ny, 0.2, U), 2
    h.set_conv_kernel(mlmc.CONV_SIMT)
    Ws = [W.astype(np.float32).astype(np.float64) for W in NN.init_weights(NN.channels_of(d, True), 9)]
    h.learned_set(np.concatenate([W.astype(np.float32).ravel() for W in Ws]), enable=0)
    R = torch.randn(nx * ny * d, k, dtype=torch.complex64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(nx + k))
    E = torch.full_like(R, float("nan"))
    h.learned_apply(R.data_ptr(), E.data_ptr(), k)
    Rn, En = R.cpu().numpy().astype(np.complex128), E.cpu().numpy()
    for c in range(0, k, 7):
        ref, _ = NN.forward(Rn[:, c], Ws, nx, ny, d, True, True)
        assert np.abs(En[:, c] - ref).max() <= 1e-5 * np.abs(ref).max()
    assert np.isfinite(En).all()
    loss, grad = h.learned_grad(R.data_ptr(), k)
    h.close()
    ref_loss, ref_g = NN.loss_and_grad(A, Rn, Ws, nx, ny, d, True, True)
    ref_flat = np.concatenate([x.ravel() for x in ref_g])
    assert abs(loss - ref_loss) <= 1e-4 * abs(ref_loss)
    assert np.abs(grad - ref_flat).max() <= 1e-3 * np.abs(ref_flat).max()
