"""Rounding of complex FP32 products: a term's product is formed first and added to the running sum,
which is rounded once per term and component."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.operators import wilson2d
from paper_2108_11281_gb300.workloads import gauge_links


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


@pytest.mark.parametrize("k", [2, 4, 7, 8])
@pytest.mark.parametrize("n", [256, 511, 1024])
def test_dense_narrow(mlmc, n, k):
    """A warp per row: chains of m = n / 32 terms and a tree of five levels.  In units of u^2 / 3 of the
    result's variance the chains add m / 2 (partial sums grow linearly in variance), each level one
    and the two roundings of the products at most one and a half, u = 2^-24."""
    g = torch.Generator(device="cuda").manual_seed(n + k)
    A = torch.randn(n, n, dtype=torch.complex64, device="cuda", generator=g)
    B = torch.randn(n, k, dtype=torch.complex64, device="cuda", generator=g)
    Y = torch.full_like(B, float("nan"))
    mlmc.dense_apply(True, A.data_ptr(), B.data_ptr(), Y.data_ptr(), n, k, mlmc.DENSE_SIMT)
    ref = A.cpu().numpy().astype(np.complex128) @ B.cpu().numpy().astype(np.complex128)
    err = np.sqrt(np.mean(np.abs(Y.cpu().numpy() - ref) ** 2) / np.mean(np.abs(ref) ** 2))
    assert err <= 2.0 ** -24 * np.sqrt((n / 64 + 6.5) / 3), err


def test_inner_solve_reaches_the_operators_rounding(mlmc):
    """24 FP32 inner steps go on until the rounding of the products A z and of the solution's update is
    all that is left of |b - A x| / |b|: the median column stops at 3.6e-7 where a sum is rounded once
    per term, at 4.6e-7 where it is rounded twice (both measured); the bound lies between."""
    N, k = 64, 32
    U = gauge_links(N, N, 0.3, 1)
    prm = mlmc.default_params(levels=3, n_tv=4, spin_split=1, setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=20,
                              coarse_sweeps=10, setup_omega=1.0, bootstrap=2, boot_iters=4, block=k, inner_its=24,
                              max_iter=1, precision=mlmc.PREC_MIXED_FP32)
    h = mlmc.Hierarchy(mlmc.OP_WILSON2D, N, N, prm, mass=-0.10, links=U)
    A = wilson2d(N, N, -0.10, U)
    b = torch.randn(A.shape[0], k, dtype=torch.complex128, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(1))
    x = torch.full_like(b, float("nan"))
    with pytest.raises(mlmc.MLMCError):
        h.solve(1, b.data_ptr(), x.data_ptr(), k, 1e-15)
    h.close()
    bn = b.cpu().numpy()
    r = np.linalg.norm(bn - A @ x.cpu().numpy(), axis=0) / np.linalg.norm(bn, axis=0)
    assert np.median(r) <= 4.1e-7, np.median(r)
