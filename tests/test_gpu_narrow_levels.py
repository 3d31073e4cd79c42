"""The Example 5.1 level's fused residual and restriction on blocks of a few columns, on both sides of the
line between one thread per aggregate and an aggregate's sites over threads (idle lanes of narrow
blocks count): P^* m (b - A x), m the sites of one colour, FP64 1e-12 of scale, FP32 1e-5; and a block of
two columns takes no longer than one of eight."""
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


@pytest.mark.parametrize("n_tv", [4, 8])
@pytest.mark.parametrize("N,k", [(256, 1), (256, 2), (256, 3), (256, 8), (192, 1), (192, 16), (128, 17), (128, 4)])
def test_restricted_residual(mlmc, N, k, n_tv):
    prm = mlmc.default_params(levels=3, n_tv=n_tv, setup_sweeps=4, coarse_sweeps=2, bootstrap=0, block=4,
                              precision=mlmc.PREC_MIXED_FP32)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, N, N, prm, shift=0.3)
    P = h.prolongation(1)
    g = torch.Generator().manual_seed(k)
    x, b = (torch.randn(N * N, k, generator=g, dtype=torch.float64) for _ in range(2))
    r = (b.numpy() - laplace2d(N, N, 0.3) @ x.numpy()).reshape(N, N, k)
    j, i = np.mgrid[0:N, 0:N]
    for colour in (0, 1):
        m = r * ((i + j) % 2 == colour)[:, :, None]
        blocks = m.reshape(N // 4, 4, N // 4, 4, k).transpose(0, 2, 1, 3, 4).reshape(-1, 16, k)
        ref = np.einsum("aiq,aik->aqk", P, blocks).reshape(-1, k)
        for prec, dt, tol in ((mlmc.PREC_FP64, torch.float64, 1e-12), (mlmc.PREC_MIXED_FP32, torch.float32, 1e-5)):
            xs, bs, rc = x.to(dt).cuda(), b.to(dt).cuda(), torch.full(ref.shape, float("nan"), dtype=dt, device="cuda")
            h.residual_restrict(1, prec, xs.data_ptr(), bs.data_ptr(), rc.data_ptr(), k, colour)
            assert np.abs(rc.cpu().numpy() - ref).max() <= tol * np.abs(ref).max(), (colour, prec)
    h.close()


def test_narrow_block_takes_no_longer(mlmc):
    """512^2 in FP64: a quarter of the data in no more time."""
    prm = mlmc.default_params(levels=4, n_tv=8, setup_sweeps=2, coarse_sweeps=2, bootstrap=0, block=8)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, 512, 512, prm)
    ms = {k: min(h.profile_kernel(9, 1, k, 20)[0] for _ in range(5)) for k in (2, 8)}
    h.close()
    assert ms[2] <= ms[8], ms
