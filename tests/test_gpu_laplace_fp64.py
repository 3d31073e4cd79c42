"""The FP64 product with the Example 5.1 operator (k_laplace_march) where its strips of four lattice
columns, walks of JB rows and 16-byte packs end: odd and narrow lattices, Dirichlet and periodic,
k = 1 (no packs) to 256.  At most five products per entry: 1e-13 of the largest."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.operators import laplace2d


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


@pytest.mark.parametrize("k", [1, 2, 5, 64, 256])
@pytest.mark.parametrize("nx,ny,periodic", [(3, 3, 0), (7, 15, 0), (63, 31, 0), (129, 5, 0), (4, 4, 1), (8, 4, 1),
                                            (12, 36, 1), (20, 8, 0)])
def test_apply(mlmc, nx, ny, periodic, k):
    kw = dict(levels=2, n_tv=1, block=4, bootstrap=0)
    if nx % 2:
        prm = mlmc.default_params(transfer=mlmc.TRANSFER_BILINEAR, **kw)
    else:
        prm = mlmc.default_params(setup_kind=mlmc.SETUP_CONSTANT, **kw)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, nx, ny, prm, shift=0.3, periodic=periodic)
    x = torch.randn(nx * ny, k, dtype=torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(nx + k))
    y = torch.full_like(x, float("nan"))
    h.apply(1, x.data_ptr(), y.data_ptr(), k)
    h.close()
    ref = laplace2d(nx, ny, 0.3, bool(periodic)) @ x.cpu().numpy()
    assert np.abs(y.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()
