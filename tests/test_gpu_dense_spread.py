"""The coarsest-level product of FP64 data and of small FP32 systems (k_dense_spread), over sizes
where its items, row groups, j slices and 16-byte rows end: n from one row to the FP32 limit of
512, k = 4 (the narrowest it takes) to ragged and wide."""
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


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,k", [(1, 4), (7, 5), (9, 32), (64, 33), (225, 48), (255, 4), (256, 128), (511, 21), (130, 3)])
def test_small_fp32_products(mlmc, cplx, n, k):
    """Within the rounding bound of an FP32 sum of n (2n) products, 2 n u |A| |B| per entry."""
    dt, wide = (torch.complex64, torch.complex128) if cplx else (torch.float32, torch.float64)
    g = torch.Generator(device="cuda").manual_seed(n + k)
    A = torch.randn(n, n, dtype=dt, device="cuda", generator=g)
    B = torch.randn(n, k, dtype=dt, device="cuda", generator=g)
    Y = torch.full_like(B, float("nan"))
    mlmc.dense_apply(cplx, A.data_ptr(), B.data_ptr(), Y.data_ptr(), n, k, which=mlmc.DENSE_SIMT)
    ref, bound = A.to(wide) @ B.to(wide), A.abs().double() @ B.abs().double()
    assert ((Y.to(wide) - ref).abs() <= (4 if cplx else 2) * (n + 1) * 2.0 ** -24 * bound).all()


@pytest.mark.parametrize("m,k", [(2, 4), (3, 21), (5, 64), (16, 64), (24, 21), (33, 7), (16, 2)])
def test_fp64_coarsest_solve(mlmc, m, k):
    """Piecewise-constant P: the coarsest operator is R A P on m^2 unknowns, and a solve there is the
    product with its inverse.  Backward stable inverse and product: error <= 100 n u cond(A_L)."""
    prm = mlmc.default_params(levels=2, n_tv=1, setup_kind=mlmc.SETUP_CONSTANT, block=k, bootstrap=0)
    h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, 4 * m, 4 * m, prm)
    p = np.kron(np.eye(m), np.full((4, 1), 0.5))
    P = np.kron(p, p)
    AL = P.T @ (laplace2d(4 * m, 4 * m) @ P)
    b = torch.randn(m * m, k, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(m))
    x = torch.full_like(b, float("nan"))
    h.solve(2, b.data_ptr(), x.data_ptr(), k, 1e-10)
    h.close()
    ref = np.linalg.solve(AL, b.cpu().numpy())
    err = np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err <= 100 * m * m * 2.0 ** -53 * np.linalg.cond(AL)
