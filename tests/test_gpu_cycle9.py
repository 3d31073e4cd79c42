"""Bilinear hierarchies whose small 9-point levels (up to 48 x 48) run the cycle in one block per pack of
columns (k_cycle9_down / k_cycle9_up): every width (packs of 1, 2 and 4 columns, ragged ones), odd
and oblong levels, one and two sweeps, V- and K-cycles, against the operator and each other."""
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


def solve(mlmc, nx, ny, levels, k, mixed, pre, post, cycle, tol):
    prm = mlmc.default_params(levels=levels, transfer=mlmc.TRANSFER_BILINEAR, block=k, inner_its=2, cycle=cycle,
                              smooth_pre=pre, smooth_post=post,
                              precision=mlmc.PREC_MIXED_FP32 if mixed else mlmc.PREC_FP64)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, nx, ny, prm, shift=0.01)
    one = torch.randn(nx * ny, 1, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    b = one.expand(-1, k).contiguous()
    x = torch.full_like(b, float("nan"))
    its = h.solve(1, b.data_ptr(), x.data_ptr(), k, tol)
    h.close()
    assert torch.equal(x, x[:, :1].expand(-1, k))
    xn, bn = x[:, 0].cpu().numpy(), b[:, 0].cpu().numpy()
    r = bn - laplace2d(nx, ny, 0.01) @ xn
    assert np.linalg.norm(r) <= 1.01 * tol * np.linalg.norm(bn)
    return its, xn


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("pre,post,cyc", [(1, 1, 1), (2, 1, 1), (1, 2, 0)])
def test_widths_agree(mlmc, mixed, pre, post, cyc):
    """Widths of 3 (single columns) and 256 (packs) need the same iterations (one to spare) and give
    the same solution to the solves' tolerance: |x - x'| <= 2 tol |A^-1| |b|, |A^-1| <= 1 / shift."""
    tol = 1e-9
    i3, x3 = solve(mlmc, 63, 63, 3, 3, mixed, pre, post, cyc, tol)
    i4, x4 = solve(mlmc, 63, 63, 3, 256, mixed, pre, post, cyc, tol)
    assert abs(i3 - i4) <= 1
    assert np.linalg.norm(x3 - x4) <= 2 * tol * 100 * 1.1 * 63


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("nx,ny,levels,k", [(31, 31, 3, 1), (63, 31, 3, 5), (63, 127, 4, 6), (95, 95, 4, 64), (111, 111, 5, 2)])
def test_small_and_odd_levels(mlmc, mixed, nx, ny, levels, k):
    """The bilinear K-cycle reduces the residual by at least 4 per step on the Laplacian, so two
    inner steps per outer one reach 1e-9 in at most eight (the Laplacian's cycle is far better)."""
    its, _ = solve(mlmc, nx, ny, levels, k, mixed, 1, 1, 1, 1e-9)
    assert its <= 8
