"""The Example 5.1 fine level at sizes where the strip-walking FP64 kernel (0.7 M entries and more) and the
one-thread-per-aggregate residual-restriction (19456 aggregate-packs and more) run: b - A x as the
restarts of a solve use it, the setup's Jacobi filter, and the restricted residual itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.hierarchy import SetupParams, build_hierarchy
from oracle.operators import laplace2d


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


@pytest.mark.parametrize("nx,ny,periodic,k", [(256, 256, 0, 16), (255, 259, 0, 11), (252, 248, 1, 13), (128, 44, 0, 200)])
def test_restarts_start_from_the_true_residual(mlmc, nx, ny, periodic, k):
    """Restarts every three steps: a wrong residual would be iterated on, or stop the solve early."""
    kw = dict(n_tv=1, block=k, bootstrap=0, fgmres_restart=3)
    if nx % 2:
        prm = mlmc.default_params(levels=3, transfer=mlmc.TRANSFER_BILINEAR, **kw)
    else:
        prm = mlmc.default_params(levels=2, setup_kind=mlmc.SETUP_CONSTANT, **kw)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, nx, ny, prm, shift=0.3, periodic=periodic)
    b = torch.randn(nx * ny, k, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(k))
    x = torch.full_like(b, float("nan"))
    its = h.solve(1, b.data_ptr(), x.data_ptr(), k, 1e-11)
    h.close()
    bn = b.cpu().numpy()
    r = np.linalg.norm(bn - laplace2d(nx, ny, 0.3, bool(periodic)) @ x.cpu().numpy(), axis=0) / np.linalg.norm(bn, axis=0)
    assert 3 < its < 60 and (r <= 1.01e-11).all(), (its, r.max())


@pytest.mark.parametrize("n_tv", [4, 8])
def test_filter_matches_oracle(mlmc, n_tv):
    """512^2 test vectors (1 M and 2 M entries): an aggregate's prolongation spans the oracle's space."""
    N = 512
    prm = mlmc.default_params(levels=4, n_tv=n_tv, setup_sweeps=6, coarse_sweeps=3, bootstrap=0, block=4)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, N, N, prm)
    lv = build_hierarchy(laplace2d(N, N), N, N, 1, SetupParams(levels=4, n_tv=n_tv, sweeps=6, coarse_sweeps=3, bootstrap=0))
    P = h.prolongation(1)
    h.close()
    Q = lv[0].P_blocks
    diff = np.abs(np.einsum("aiq,ajq->aij", P, P) - np.einsum("aiq,ajq->aij", Q, Q)).max()
    assert diff <= 1e-9, diff


@pytest.mark.parametrize("nx,ny,periodic,k", [(256, 256, 0, 16), (256, 256, 1, 41), (512, 128, 0, 10), (256, 264, 0, 40)])
def test_restricted_residual(mlmc, nx, ny, periodic, k):
    """P^* m (b - A x), m the sites of one colour: FP64 1e-12 of scale, FP32 1e-5."""
    prm = mlmc.default_params(levels=3, n_tv=4, setup_sweeps=4, coarse_sweeps=2, bootstrap=0, block=4, agg_y=2 if ny == 264 else 4,
                              precision=mlmc.PREC_MIXED_FP32)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, nx, ny, prm, shift=0.3, periodic=periodic)
    P, ay = h.prolongation(1), prm.agg_y
    g = torch.Generator().manual_seed(k)
    x, b = (torch.randn(nx * ny, k, generator=g, dtype=torch.float64) for _ in range(2))
    r = (b.numpy() - laplace2d(nx, ny, 0.3, bool(periodic)) @ x.numpy()).reshape(ny, nx, k)
    j, i = np.mgrid[0:ny, 0:nx]
    for colour in (0, 1):
        m = r * ((i + j) % 2 == colour)[:, :, None]
        blocks = m.reshape(ny // ay, ay, nx // 4, 4, k).transpose(0, 2, 1, 3, 4).reshape(-1, 4 * ay, k)
        ref = np.einsum("aiq,aik->aqk", P, blocks).reshape(-1, k)
        for prec, dt, tol in ((mlmc.PREC_FP64, torch.float64, 1e-12), (mlmc.PREC_MIXED_FP32, torch.float32, 1e-5)):
            xs, bs, rc = x.to(dt).cuda(), b.to(dt).cuda(), torch.full(ref.shape, float("nan"), dtype=dt, device="cuda")
            h.residual_restrict(1, prec, xs.data_ptr(), bs.data_ptr(), rc.data_ptr(), k, colour)
            assert np.abs(rc.cpu().numpy() - ref).max() <= tol * np.abs(ref).max(), (colour, prec)
    h.close()
