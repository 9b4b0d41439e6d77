"""FP64 batches and the tiled passes (k_tiles64.cu): which images take them, and groups of every size beside a largest
one of 8 or 16, whose layout they share (with 16, a group of 1 has more lanes than a tile has pixels)."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads.configs import ct_op
from workloads.problem import Problem, RegDesc, SketchDesc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


def solves(G, N, views, count):
    """Iterates with the tiles where the rule takes them, and on the row kernels; the problems."""
    A = ct_op(N, np.arange(views) * 180.0 / views, int(1.43 * N) + 1)
    assert A.val.size >= 1 << 20
    M = (A.row_ptr, A.col, A.val.astype(np.float64))
    rng = np.random.default_rng(count)
    probs = []
    for i in range(count):
        x = rng.uniform(0.0, 1.0, A.n).astype(np.float32).astype(np.float64)
        b = np.add.reduceat(np.append(M[2] * x[M[1]], 0.0), M[0][:-1]) * (np.diff(M[0]) > 0)
        b = (b * (1.0 + 0.02 * rng.standard_normal(A.m))).astype(np.float32).astype(np.float64)
        probs.append(Problem("t", A, RegDesc("grad2d", nx=N, ny=N), b, x, 10.0 ** rng.uniform(0, 1), 4,
                             SketchDesc("sparse_sign", 60, 8, 3)))
    kw = G.device_inputs(probs[0], "fp64")
    insts = [dict(A=kw["A"], reg=kw["reg"], lam=P.lam, b=torch.from_numpy(P.b).cuda()) for P in probs]
    xs = []
    for tiles in (True, False):
        Bt = G.Batch(insts, 60, 3, max_iters=4, precision="fp64", tiles=tiles)
        Bt.solve(4)
        xs.append(Bt.x())
        Bt.close()
    return xs, probs


@pytest.mark.parametrize("N,views,count,tiled", [(80, 150, 2, False), (97, 100, 4, False), (160, 40, 8, False),
                                                 (64, 240, 16, False), (112, 80, 16, False), (192, 40, 2, True),
                                                 (192, 40, 8, True), (128, 60, 16, True)])
def test_images_that_take_the_tiles(G, N, views, count, tiled):
    """Fewer CTAs than the rule of build_tiles64 wants: the row kernels, bit for bit."""
    xs, _ = solves(G, N, views, count)
    assert all(torch.equal(a, b) for a, b in zip(*xs)) != tiled


@pytest.mark.parametrize("count", [11, 13, 17, 18, 20, 23])
def test_groups_beside_a_larger_one(G, count):
    xs, probs = solves(G, 192, 40, count)
    for i, P in enumerate(probs):
        ref = torch.from_numpy(O.sgks(P)["x"]).cuda() if i in (0, count - 1) else xs[1][i]
        for x in (xs[0][i], xs[1][i]):
            assert torch.linalg.norm(x - ref) <= 1e-10 * torch.linalg.norm(ref)
