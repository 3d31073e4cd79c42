"""The cycle's fused residual and restriction on levels with eight coarse dofs (FP32 data), over even
and odd aggregates, 2 -> 8 and 8 -> 8 dofs, real and complex, ragged column counts.  The FP64 form
runs the same cycle with a residual and a restriction kernel of their own, so both need the same
outer iterations for a tolerance well above FP32's (one to spare)."""
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


@pytest.mark.parametrize("op,nx,ny,agg,levels,k", [("wilson", 32, 32, 4, 3, 32), ("wilson", 36, 36, 3, 3, 7),
                                                   ("wilson", 24, 24, 3, 2, 33), ("wilson", 16, 8, 2, 3, 1),
                                                   ("laplace", 64, 32, 4, 3, 33), ("laplace", 36, 36, 3, 3, 5)])
def test_same_iterations_as_separate_kernels(mlmc, op, nx, ny, agg, levels, k):
    its = []
    for precision in (mlmc.PREC_FP64, mlmc.PREC_MIXED_FP32):
        kw = dict(levels=levels, agg_x=agg, agg_y=agg, block=k, inner_its=2, bootstrap=0, precision=precision)
        if op == "wilson":
            U = gauge_links(nx, ny, 0.3, 2)
            prm = mlmc.default_params(n_tv=4, spin_split=1, setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=6,
                                      setup_omega=1.0, **kw)
            h = mlmc.Hierarchy(mlmc.OP_WILSON2D, nx, ny, prm, mass=0.1, links=U)
            A, dt = wilson2d(nx, ny, 0.1, U), torch.complex128
        else:
            h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, nx, ny, mlmc.default_params(n_tv=8, setup_sweeps=10, **kw))
            A, dt = laplace2d(nx, ny), torch.float64
        b = torch.randn(A.shape[0], k, dtype=dt, device="cuda", generator=torch.Generator(device="cuda").manual_seed(k))
        x = torch.full_like(b, float("nan"))
        its.append(h.solve(1, b.data_ptr(), x.data_ptr(), k, 1e-7))
        h.close()
        bn = b.cpu().numpy()
        res = np.linalg.norm(bn - A @ x.cpu().numpy(), axis=0) / np.linalg.norm(bn, axis=0)
        assert res.max() <= 1e-7
    assert abs(its[0] - its[1]) <= 1, its
