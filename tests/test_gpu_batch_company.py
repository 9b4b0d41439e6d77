"""An instance's result depends on the group it is in, not on how many other groups the batch has."""
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


# 97^2 is too small for the FP64 tiled passes, 192^2 takes them
@pytest.mark.parametrize("count,prec,N", [(2, "ff", 97), (16, "ff", 97), (16, "fp32", 97), (4, "fp64", 97),
                                          (4, "fp64", 192), (16, "fp64", 192)])
def test_another_group_changes_no_bits(G, count, prec, N):
    A = ct_op(N, np.arange(40) * 4.5, int(1.43 * N) + 1)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    C = G.CSR(dev(A.row_ptr), dev(A.col), dev(A.val.astype(np.float32)), A.m, A.n).transposed()
    g = torch.Generator(device="cuda").manual_seed(2)
    bs = [torch.rand(A.m, generator=g, device="cuda", dtype=torch.float64).to(G.io_dtype(prec)) for _ in range(count + 1)]
    xs = []
    for k in (count, count + 1):   # one group, and the same group with another one beside it
        Bt = G.Batch([dict(A=C, reg=G.Reg("grad2d", N, N), lam=2.0, b=b) for b in bs[:k]], 60, 3, max_iters=5,
                     precision=prec)
        Bt.solve(5)
        xs.append(Bt.x())
        Bt.close()
    assert all(torch.equal(a, b) for a, b in zip(*xs))
