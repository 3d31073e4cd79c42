"""The fixed-length FGMRES where its last step brings nothing new: a two-grid cycle without smoothing on one
aggregate has rank one, so every preconditioned vector is a multiple of P, A z of the second step lies
in the span of the first, and the second step's minimum is the first's.  What the last diagonal entry
holds is then rounding, and must not become a coefficient: the residual after two steps is that after
one, to 1e-6 of |b| in FP64 (square root of the rounding) and 1e-3 in FP32."""
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


def residual(mlmc, op, N, k, inner, mixed, b):
    kw = dict(levels=2, agg_x=N, agg_y=N, n_tv=1, block=k, bootstrap=0, smooth_pre=0, smooth_post=0, inner_its=inner,
              max_iter=1, precision=mlmc.PREC_MIXED_FP32 if mixed else mlmc.PREC_FP64)
    if op == "laplace":
        h = mlmc.Hierarchy(mlmc.OP_LAPLACE2D, N, N, mlmc.default_params(setup_kind=mlmc.SETUP_CONSTANT, **kw))
        A = laplace2d(N, N)
    else:
        U = gauge_links(N, N, 0.3, 2)
        h = mlmc.Hierarchy(mlmc.OP_WILSON2D, N, N, mlmc.default_params(setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=4,
                                                                      setup_omega=1.0, **kw), mass=0.1, links=U)
        A = wilson2d(N, N, 0.1, U)
    x = torch.full_like(b, float("nan"))
    with pytest.raises(mlmc.MLMCError):
        h.solve(1, b.data_ptr(), x.data_ptr(), k, 1e-15)
    h.close()
    bn = b.cpu().numpy()
    return np.linalg.norm(bn - A @ x.cpu().numpy(), axis=0) / np.linalg.norm(bn, axis=0)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("op,N,k", [("laplace", 16, 64), ("laplace", 32, 33), ("wilson", 8, 32)])
def test_a_redundant_last_step_changes_nothing(mlmc, op, N, k, mixed):
    n = N * N * (2 if op == "wilson" else 1)
    b = torch.randn(n, k, dtype=torch.complex128 if op == "wilson" else torch.float64, device="cuda",
                    generator=torch.Generator(device="cuda").manual_seed(5))
    one = residual(mlmc, op, N, k, 1, mixed, b)
    two = residual(mlmc, op, N, k, 2, mixed, b)
    assert (one < 1.0).all()
    assert (two <= one + (1e-3 if mixed else 1e-6)).all(), (two - one).max()
