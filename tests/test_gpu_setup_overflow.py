"""A start vector whose norm overflows has an infinite norm, not NaN (k_setup.cu, norms with their rounding errors
added): A^T b / ||A^T b|| is then 0 and the solve reports a breakdown."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


@pytest.mark.parametrize("method", ["sgks", "gks"])
def test_infinite_norm_of_the_start_vector(G, method):
    n = 40
    A = G.Conv2D(torch.full((3, 3), 1.0 / 9.0, device="cuda"), n, n)
    g = torch.Generator(device="cuda").manual_seed(0)
    b = torch.rand(n * n, generator=g, device="cuda", dtype=torch.float64) * 1e200
    S = G.Solver(A, G.Reg("grad2d", n, n), b, 0.1, 60, 3, max_iters=4, method=method)
    assert S.status() == 1     # SGKS_BREAKDOWN
    S.close()
