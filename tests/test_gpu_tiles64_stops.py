"""Instances of an FP64 batch that stop at different iterations (eq. RC), on the tiled passes (k_tiles64.cu): a CTA
then holds live and stopped instances.  The same stops and iterates as on the row kernels."""
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


@pytest.mark.parametrize("count", [8, 16])
def test_early_stops(G, count):
    A = ct_op(192, np.arange(40) * 4.5, 275)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    C = G.CSR(dev(A.row_ptr), dev(A.col), dev(A.val.astype(np.float32)), A.m, A.n).transposed()
    rng = np.random.default_rng(count)
    # lambda from heavy regularization, which settles early, to little of it
    insts = [dict(A=C, reg=G.Reg("grad2d", 192, 192), lam=10.0 ** (3.0 - 5.0 * i / (count - 1)),
                  b=dev(rng.uniform(0.5, 1.5, A.m))) for i in range(count)]
    runs = []
    for tiles in (True, False):
        Bt = G.Batch(insts, 60, 3, max_iters=12, precision="fp64", tiles=tiles)
        reps = Bt.solve(12, tol=3e-2)
        runs.append(([r["iters_done"] for r in reps], [r["status"] for r in reps], Bt.x()))
        Bt.close()
    assert runs[0][:2] == runs[1][:2]
    assert len(set(runs[0][0])) > 2, runs[0][0]
    for x, r in zip(runs[0][2], runs[1][2]):
        assert torch.linalg.norm(x - r) <= 1e-10 * torch.linalg.norm(r)
