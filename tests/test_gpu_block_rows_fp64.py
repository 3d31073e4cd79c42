"""Products with real 8 x 8 block stencils in FP64 on both sides of one block per SM, where the
coefficients go through shared memory or through the cache: 64 to 1024 sites, one column to 130.  The
blocks are read back from the library; 40 products per entry: 1e-13 of the largest."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


@pytest.mark.parametrize("nx,ny", [(32, 32), (48, 48), (64, 64), (128, 128), (64, 24)])
def test_apply(mlmc, nx, ny):
    prm = mlmc.default_params(levels=2, n_tv=8, setup_sweeps=6, bootstrap=0, block=4)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, nx, ny, prm, shift=0.1)
    cx, cy, d = h.level_info(2)
    A = h.operator(2).reshape(cy, cx, 5, d, d)
    for k in (1, 5, 31, 33, 64, 66, 100, 130):
        x = torch.randn(cx * cy * d, k, dtype=torch.float64, device="cuda",
                        generator=torch.Generator(device="cuda").manual_seed(k))
        y = torch.full_like(x, float("nan"))
        h.apply(2, x.data_ptr(), y.data_ptr(), k)
        X = x.cpu().numpy().reshape(cy, cx, d, k)
        nbs = (X, np.roll(X, -1, 1), np.roll(X, 1, 1), np.roll(X, -1, 0), np.roll(X, 1, 0))
        ref = sum(np.einsum("jirq,jiqk->jirk", A[:, :, t], v) for t, v in enumerate(nbs))
        err = np.abs(y.cpu().numpy().reshape(ref.shape) - ref).max()
        assert err <= 1e-13 * np.abs(ref).max(), (k, err)
    h.close()
