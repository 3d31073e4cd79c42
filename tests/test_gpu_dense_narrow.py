"""FP32 dense products of four to eight columns (the CUDA-core route): a warp per row from n = 512 on,
spread slices below.  A sum of n / 32 terms per lane and a tree of five levels rounds with a
variance of at most (n / 64 + 5) u^2 / 3 of the result's (partial sums grow linearly in
variance), u = 2^-24, so the rms error stays below u sqrt((n / 64 + 5) / 3)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mlmc():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2108_11281_gb300 import mlmc as m
    return m


@pytest.mark.parametrize("k", [4, 5, 8])
@pytest.mark.parametrize("n", [100, 256, 511, 512, 577, 1024, 2048])
def test_rounding_is_that_of_short_sums(mlmc, n, k):
    g = torch.Generator(device="cuda").manual_seed(n + k)
    A = torch.randn(n, n, dtype=torch.float32, device="cuda", generator=g)
    B = torch.randn(n, k, dtype=torch.float32, device="cuda", generator=g)
    Y = torch.full_like(B, float("nan"))
    mlmc.dense_apply(False, A.data_ptr(), B.data_ptr(), Y.data_ptr(), n, k, mlmc.DENSE_SIMT)
    ref = A.cpu().numpy().astype(np.float64) @ B.cpu().numpy().astype(np.float64)
    err = np.sqrt(np.mean((Y.cpu().numpy() - ref) ** 2) / np.mean(ref ** 2))
    assert err <= 2.0 ** -24 * np.sqrt((n / 64 + 5) / 3), err
