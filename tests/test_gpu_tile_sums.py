"""Rounding of the tiled transposed pass (k_tiles.cu): a pixel's entries are added on one lane where the row kernel
has eight, in a tree that is to lose no more.  Emulated in numpy for rows of 36 to 240 entries of one or both signs, cut
into stages as here, the tree's rms error is 0.5 to 1.2 times that of the row kernel's order; hence 1.25 for the
errors of x after one iteration, which both come from the same sums (blocks of 16 terms one after the other: 1.3 to 1.8)."""
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


@pytest.mark.parametrize("N,views,count", [(97, 100, 2), (181, 180, 1), (181, 180, 2), (181, 180, 16), (256, 30, 2),
                                           (256, 30, 16)])
def test_error_against_the_row_kernels(G, N, views, count):
    A = ct_op(N, np.arange(views) * 180.0 / views, int(1.43 * N) + 1)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    C = G.CSR(dev(A.row_ptr), dev(A.col), dev(A.val.astype(np.float32)), A.m, A.n).transposed()
    sq = dict(tiles=0.0, rows=0.0)
    for seed in range(6):
        g = torch.Generator(device="cuda").manual_seed(seed)
        bs = [torch.rand(A.m, generator=g, device="cuda").double() for _ in range(count)]
        x = {}
        for name, prec, tiles in (("ref", "fp64", False), ("tiles", "ff", True), ("rows", "ff", False)):
            Bt = G.Batch([dict(A=C, reg=G.Reg("grad2d", N, N), lam=5.0, b=b) for b in bs], 200, 3, max_iters=1,
                         precision=prec, tiles=tiles)
            Bt.solve(1)
            x[name] = torch.stack(Bt.x())
            Bt.close()
        for k in sq:
            sq[k] += float(torch.sum((x[k] - x["ref"]) ** 2))
    assert sq["tiles"] <= 1.25**2 * sq["rows"]
