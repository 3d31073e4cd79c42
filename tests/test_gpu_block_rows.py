"""The row-split block stencil and smoother (d = 8 dofs per site) over block widths where their
column groups end: one column per thread and two (even widths from 64 on), full and ragged
warps.  Columns are independent systems that take the same operations in the same order, so
equal right-hand sides give bitwise equal solutions, and the iteration count does not depend on
the width (by more than the one that the different grouping of the dot products may cost)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2108_11281_gb300.workloads import gauge_links

WIDTHS = [1, 3, 32, 33, 64, 65, 66, 130]


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


def make(mlmc, op, k, mixed):
    kw = dict(levels=3, block=k, inner_its=4, smooth_pre=2, smooth_post=2, bootstrap=0,
              precision=mlmc.PREC_MIXED_FP32 if mixed else mlmc.PREC_FP64)
    if op == "laplace":
        return mlmc.Hierarchy(mlmc.OP_LAPLACE2D, 64, 32, mlmc.default_params(n_tv=8, setup_sweeps=20, **kw))
    prm = mlmc.default_params(n_tv=4, spin_split=1, setup_kind=mlmc.SETUP_INVERSE, setup_sweeps=6, setup_omega=1.0, **kw)
    return mlmc.Hierarchy(mlmc.OP_WILSON2D, 32, 64, prm, mass=0.1, links=gauge_links(32, 64, 0.3, 2))


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("op", ["laplace", "wilson"])
def test_equal_columns(mlmc, op, mixed):
    its = []
    for k in WIDTHS:
        h = make(mlmc, op, k, mixed)
        assert h.level_info(2)[2] == 8
        dt = torch.complex128 if op == "wilson" else torch.float64
        one = torch.randn(h.n(2), 1, dtype=dt, device="cuda", generator=torch.Generator(device="cuda").manual_seed(4))
        b = one.expand(-1, k).contiguous()
        x = torch.full_like(b, float("nan"))
        its.append(h.solve(2, b.data_ptr(), x.data_ptr(), k, 1e-10))
        r = torch.empty_like(x)
        h.apply(2, x.data_ptr(), r.data_ptr(), k)
        h.close()
        assert torch.equal(x, x[:, :1].expand(-1, k))
        assert float(torch.linalg.norm(b[:, 0] - r[:, 0]) / torch.linalg.norm(b[:, 0])) <= 1.01e-10
    assert max(its) - min(its) <= 1, its
