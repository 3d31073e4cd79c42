"""The fixed-length FGMRES inside the level solves (partial dots, their per-column algebra, the
multi-AXPY and the last step's least-squares problem) over the lengths and block widths where
its kernels change form: one step (first and last at once), the last single pass over the basis
(8 vectors), several passes (9, 32); widths below and above a 16-byte pack, ragged ones, and
widths whose columns do not divide the 512 threads of a block."""
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


def make(mlmc, op, N, k, inner, mixed, **kw):
    kw = dict(dict(levels=2, block=k, inner_its=inner, precision=mlmc.PREC_MIXED_FP32 if mixed else mlmc.PREC_FP64,
                   fgmres_restart=32), **kw)
    if op == "laplace":
        prm = mlmc.default_params(n_tv=4, setup_sweeps=20, bootstrap=0, **kw)
        return mlmc.Hierarchy(mlmc.OP_LAPLACE2D, N, N, prm), laplace2d(N, N), torch.float64
    U = gauge_links(N, N, 0.3, 2)
    prm = mlmc.default_params(n_tv=2, spin_split=1, setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=4, setup_omega=1.0,
                              bootstrap=0, **kw)
    return mlmc.Hierarchy(mlmc.OP_WILSON2D, N, N, prm, mass=0.1, links=U), wilson2d(N, N, 0.1, U), torch.complex128


def iterate(mlmc, h, b, k):
    """The iterate that a solve with a small max_iter ends on (status: not converged)."""
    x = torch.full_like(b, float("nan"))
    try:
        h.solve(1, b.data_ptr(), x.data_ptr(), k, 1e-15)
    except mlmc.MLMCError as e:
        assert e.status == mlmc.ERR_NOT_CONVERGED
    h.close()
    return x.cpu().numpy()


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("op", ["laplace", "wilson"])
@pytest.mark.parametrize("inner,k", [(1, 1), (2, 3), (8, 4), (8, 12), (9, 21), (32, 64), (2, 200)])
def test_inner_lengths_and_widths(mlmc, op, mixed, inner, k):
    """One outer step around `inner` inner steps and `inner` steps of the restarted solver (the
    textbook form with a normalised FP64 basis) both minimise the residual over the same Krylov
    space of the two-level cycle, so their residuals agree column by column: to 1e-6 in FP64, and
    in the mixed form, whose inner basis is FP32, to 1e-2 above FP32's own level of 1e-5."""
    N = 16
    h, A, dt = make(mlmc, op, N, k, inner, mixed, max_iter=1)
    b = torch.randn(A.shape[0], k, dtype=dt, device="cuda", generator=torch.Generator(device="cuda").manual_seed(k))
    x = iterate(mlmc, h, b, k)
    h, _, _ = make(mlmc, op, N, k, 0, mixed, max_iter=inner)
    ref = iterate(mlmc, h, b, k)
    bn = b.cpu().numpy()
    norm = np.linalg.norm(bn, axis=0)
    r, r0 = (np.linalg.norm(bn - A @ v, axis=0) / norm for v in (x, ref))
    rtol, atol = (1e-2, 1e-5) if mixed else (1e-6, 1e-12)
    assert (np.abs(r - r0) <= rtol * r0 + atol).all(), np.abs(r - r0).max()


def test_zero_columns_stay_zero(mlmc):
    """A zero right-hand side among others: its column is never iterated and solves to zero."""
    h, A, dt = make(mlmc, "laplace", 16, 5, 8, True)
    b = torch.randn(A.shape[0], 5, dtype=dt, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    b[:, 2] = 0.0
    x = torch.full_like(b, float("nan"))
    h.solve(1, b.data_ptr(), x.data_ptr(), 5, 1e-10)
    h.close()
    assert torch.count_nonzero(x[:, 2]) == 0
    r = b.cpu().numpy() - A @ x.cpu().numpy()
    live = [0, 1, 3, 4]
    assert (np.linalg.norm(r[:, live], axis=0) <= 1e-10 * np.linalg.norm(b.cpu().numpy()[:, live], axis=0)).all()
