"""Data beyond the range of the FP64 tiled passes (k_tiles64.cu: exact up to 2^575) end a solve as on the row kernels:
the squared norms overflow, A^T b / ||A^T b|| is 0, and that is a breakdown."""
import numpy as np
import pytest
import torch

from workloads.configs import ct_op

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


@pytest.mark.parametrize("scale", [1e160, 1e200, 1e300])
def test_large_data(G, scale):
    A = ct_op(192, np.arange(40) * 4.5, 275)
    assert A.val.size >= 1 << 20
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    C = G.CSR(dev(A.row_ptr), dev(A.col), dev(A.val.astype(np.float32)), A.m, A.n).transposed()
    rng = np.random.default_rng(1)
    b, plain = dev(rng.uniform(0.5, 1.5, A.m)) * scale, dev(rng.uniform(0.5, 1.5, A.m))
    reg = G.Reg("grad2d", 192, 192)
    S = G.Solver(C, reg, b, 1.0, 60, 3, max_iters=4)
    assert S.status() == 1     # SGKS_BREAKDOWN
    S.close()
    xs = []
    for tiles in (True, False):
        Bt = G.Batch([dict(A=C, reg=reg, lam=1.0, b=v) for v in (b, plain)], 60, 3, max_iters=4, tiles=tiles)
        Bt.solve(4)
        assert Bt.status() == [1, 0]
        xs.append(Bt.x()[1])
        Bt.close()
    assert torch.linalg.norm(xs[0] - xs[1]) <= 1e-10 * torch.linalg.norm(xs[1])
