"""One multigrid cycle against the oracle's, column by column.  A solve of one outer step without inner
steps returns x = a z with z the cycle's result for b and a the minimiser of |b - a A z|, so its
kernels (the first smoother sweep from zero, fused residual and restriction, prolongation over
dofs, the bilinear levels' two-launch cycle) show in x itself, where a converged solve would correct
them.  FP64: 1e-9 of the largest entry.  Mixed form: a cycle in FP32 rounds some hundred times (u =
6e-8) and its coarsest inverse has a condition below 1e3: 5e-4."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.bilinear import build_bilinear_hierarchy
from oracle.hierarchy import SetupParams, build_hierarchy
from oracle.operators import laplace2d, wilson2d
from oracle.solver import Cycle
from paper_2108_11281_gb300.workloads import gauge_links


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


def check(mlmc, make, lv, k, smooth, cycle, cplx, levels=(1,)):
    kw = dict(block=k, coarse_block=k, bootstrap=0, inner_its=0, max_iter=1, fgmres_restart=1, smooth_pre=smooth[0],
              smooth_post=smooth[1], cycle=mlmc.CYCLE_K if cycle == "K" else mlmc.CYCLE_V)
    cols = sorted({0, k // 2, k - 1})
    for mixed in (0, 1):
        h = make(precision=mlmc.PREC_MIXED_FP32 if mixed else mlmc.PREC_FP64, **kw)
        for level in levels:
            A = lv[level - 1].A
            b = torch.randn(A.shape[0], k, dtype=torch.complex128 if cplx else torch.float64, device="cuda",
                            generator=torch.Generator(device="cuda").manual_seed(k + level))
            x = torch.full_like(b, float("nan"))
            with pytest.raises(mlmc.MLMCError) as e:
                h.solve(level, b.data_ptr(), x.data_ptr(), k, 1e-15)
            assert e.value.status == mlmc.ERR_NOT_CONVERGED
            ref_cycle = Cycle(lv, first=level - 1, pre=smooth[0], post=smooth[1], kind=cycle, kcycle_its=2)
            xn, bn = x.cpu().numpy(), b.cpu().numpy()
            assert np.isfinite(xn).all()
            for c in cols:
                z = ref_cycle(bn[:, c])
                Az = A @ z
                ref = z * (np.vdot(Az, bn[:, c]) / np.vdot(Az, Az).real)
                err = np.abs(xn[:, c] - ref).max() / np.abs(ref).max()
                assert err <= (5e-4 if mixed else 1e-9), (mixed, level, c, err)
        h.close()


@pytest.mark.parametrize("N,agg,levels,n_tv,k,smooth,cycle", [
    (64, 4, 3, 4, 5, (2, 2), "K"), (64, 4, 3, 4, 33, (2, 1), "V"), (256, 4, 4, 4, 32, (3, 1), "V"),
    (256, 4, 3, 4, 40, (1, 1), "V"), (64, 4, 3, 8, 33, (2, 2), "K"), (64, 4, 3, 8, 64, (3, 2), "V"), (36, 3, 3, 8, 7, (2, 1), "K"),
    (36, 3, 3, 2, 6, (2, 2), "K"), (64, 4, 3, 1, 16, (2, 1), "K")])
def test_laplacian(mlmc, N, agg, levels, n_tv, k, smooth, cycle):
    A = laplace2d(N, N, 0.1)
    if n_tv == 1:
        sp = SetupParams(levels=levels, agg_x=agg, agg_y=agg, n_tv=1, kind="constant", bootstrap=0)
    else:
        sp = SetupParams(levels=levels, agg_x=agg, agg_y=agg, n_tv=n_tv, sweeps=10, coarse_sweeps=5, bootstrap=0)
    lv = build_hierarchy(A, N, N, 1, sp)

    def make(**kw):
        prm = mlmc.default_params(levels=levels, agg_x=agg, agg_y=agg, n_tv=n_tv, **kw)
        return mlmc.Hierarchy(mlmc.OP_LAPLACE2D, N, N, prm, shift=0.1, user_P=[v.P_blocks for v in lv[:-1]])
    check(mlmc, make, lv, k, smooth, cycle, False, levels=(1, 2) if levels > 2 else (1,))


@pytest.mark.parametrize("N,agg,levels,n_tv,k,smooth,cycle", [
    (32, 4, 3, 4, 32, (2, 2), "K"), (32, 4, 3, 4, 66, (2, 1), "V"), (32, 4, 2, 4, 5, (3, 1), "V"), (36, 3, 3, 4, 7, (2, 2), "K"),
    (32, 4, 3, 2, 33, (2, 1), "K"), (16, 2, 3, 2, 64, (1, 1), "V")])
def test_wilson(mlmc, N, agg, levels, n_tv, k, smooth, cycle):
    U = gauge_links(N, N, 0.3, 5)
    A = wilson2d(N, N, 0.2, U)
    lv = build_hierarchy(A, N, N, 2, SetupParams(levels=levels, agg_x=agg, agg_y=agg, n_tv=n_tv, spin_split=True,
                                                 kind="inverse", sweeps=4, coarse_sweeps=4, omega=1.0, noise_kind="z4",
                                                 bootstrap=0))

    def make(**kw):
        prm = mlmc.default_params(levels=levels, agg_x=agg, agg_y=agg, n_tv=n_tv, spin_split=1, **kw)
        return mlmc.Hierarchy(mlmc.OP_WILSON2D, N, N, prm, mass=0.2, links=U, user_P=[v.P_blocks for v in lv[:-1]])
    check(mlmc, make, lv, k, smooth, cycle, True, levels=(1, 2) if levels > 2 else (1,))


@pytest.mark.parametrize("N,levels,k,smooth,cycle", [(63, 4, 5, (1, 1), "K"), (63, 3, 256, (2, 1), "V"), (95, 4, 1, (1, 2), "K"),
                                                     (95, 3, 8, (2, 2), "V"), (127, 3, 6, (1, 1), "V"), (31, 3, 200, (1, 1), "K")])
def test_bilinear(mlmc, N, levels, k, smooth, cycle):
    lv = build_bilinear_hierarchy(N, levels, 0.1)

    def make(**kw):
        prm = mlmc.default_params(levels=levels, transfer=mlmc.TRANSFER_BILINEAR, **kw)
        return mlmc.Hierarchy(mlmc.OP_LAPLACE2D, N, N, prm, shift=0.1)
    check(mlmc, make, lv, k, smooth, cycle, False, levels=(1, 2))
