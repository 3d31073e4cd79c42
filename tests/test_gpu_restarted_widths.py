"""The restarted FGMRES with the library's default parameters (no inner solve, up to 30 basis vectors
per cycle) over block widths: one column, packs and ragged ones, widths that the 512 threads of a
block do not divide, and 256, whose multi-AXPY coefficients take more than one pass.  A column's
iterates do not depend on the others, so equal right-hand sides take the same steps at any width."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

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


def make(mlmc, op, N, k, **kw):
    if op == "laplace":
        prm = mlmc.default_params(n_tv=1, setup_kind=mlmc.SETUP_CONSTANT, block=k, bootstrap=0, **kw)
        return mlmc.Hierarchy(mlmc.OP_LAPLACE2D, N, N, prm), laplace2d(N, N), torch.float64
    U = gauge_links(N, N, 0.3, 2)
    prm = mlmc.default_params(n_tv=2, spin_split=1, setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=4, setup_omega=1.0,
                              block=k, bootstrap=0, **kw)
    return mlmc.Hierarchy(mlmc.OP_WILSON2D, N, N, prm, mass=0.1, links=U), wilson2d(N, N, 0.1, U), torch.complex128


@pytest.mark.parametrize("reorth", [0, 1])
@pytest.mark.parametrize("op", ["laplace", "wilson"])
def test_equal_columns_take_the_same_steps(mlmc, op, reorth):
    """Iterations agree to one step and every column reaches the tolerance, at all widths."""
    tol, its = 1e-10, {}
    for k in (1, 2, 3, 8, 21, 62, 200, 256):
        h, A, dt = make(mlmc, op, 32, k, reorth=reorth)
        one = torch.randn(A.shape[0], 1, dtype=dt, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
        b = one.expand(-1, k).contiguous()
        x = torch.full_like(b, float("nan"))
        its[k] = h.solve(1, b.data_ptr(), x.data_ptr(), k, tol)
        h.close()
        bn = b.cpu().numpy()
        r = np.linalg.norm(bn - A @ x.cpu().numpy(), axis=0) / np.linalg.norm(bn, axis=0)
        assert (r <= 1.01 * tol).all(), (k, r.max())
    assert max(its.values()) - min(its.values()) <= 1 and min(its.values()) > 8, its


def test_one_column_takes_no_longer_than_a_wide_block(mlmc):
    """The same 64^2 solve (23 steps or more, so up to 23 basis vectors per reduction) with 1 / 200 of the
    data: its reductions are shorter chains, not longer ones."""
    import time
    best = {}
    for k in (1, 200):
        h, A, dt = make(mlmc, "laplace", 64, k)
        b = torch.randn(A.shape[0], k, dtype=dt, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
        x = torch.empty_like(b)
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            h.solve(1, b.data_ptr(), x.data_ptr(), k, 1e-10)
            best[k] = min(best.get(k, 1e9), time.perf_counter() - t)
        h.close()
    assert best[1] <= best[200], best
