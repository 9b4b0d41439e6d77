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


@pytest.mark.parametrize("count,prec", [(2, "ff"), (16, "ff"), (16, "fp32"), (4, "fp64"), (16, "fp64")])
def test_another_group_changes_no_bits(G, count, prec):
    A = ct_op(97, np.arange(100) * 1.8, 139)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    C = G.CSR(dev(A.row_ptr), dev(A.col), dev(A.val.astype(np.float32)), A.m, A.n).transposed()
    g = torch.Generator(device="cuda").manual_seed(2)
    bs = [torch.rand(A.m, generator=g, device="cuda", dtype=torch.float64).to(G.io_dtype(prec)) for _ in range(count + 1)]
    xs = []
    for k in (count, count + 1):   # one group, and the same group with another one beside it
        Bt = G.Batch([dict(A=C, reg=G.Reg("grad2d", 97, 97), lam=2.0, b=b) for b in bs[:k]], 60, 3, max_iters=5,
                     precision=prec)
        Bt.solve(5)
        xs.append(Bt.x())
        Bt.close()
    assert all(torch.equal(a, b) for a, b in zip(*xs))
