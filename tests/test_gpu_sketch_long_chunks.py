"""Column chunks of the compensated batches' sketches (k_sketchx.cu) at the lengths that vectors of more than 77,824
values have: 448 columns, and the longest ones, 1,024 and, with 16 instances, 768 (98 KB of shared memory).  Compared
with the oracle at the float-float bar, 1e-10."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads.configs import conv2d_op, gaussian_psf
from workloads.problem import Problem, RegDesc, SketchDesc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


@pytest.mark.parametrize("nx,ny,count", [(213, 212, 1), (213, 212, 8), (331, 320, 1), (331, 320, 8), (331, 320, 16)])
def test_long_chunks(G, nx, ny, count):
    A, L = conv2d_op(nx, ny, gaussian_psf(5, 1.2)), RegDesc("grad2d", nx=nx, ny=ny)
    rng = np.random.default_rng(nx + count)
    probs = []
    for i in range(count):
        x = rng.uniform(0.0, 1.0, A.n).astype(np.float32).astype(np.float64)
        b = (x * (1.0 + 0.02 * rng.standard_normal(A.m))).astype(np.float32).astype(np.float64)
        probs.append(Problem("t", A, L, b, x, 10.0 ** rng.uniform(-2, 0), 4, SketchDesc("sparse_sign", 61, 8, 5)))
    kw = G.device_inputs(probs[0], "ff")
    Bt = G.Batch([dict(A=kw["A"], reg=kw["reg"], lam=P.lam, b=torch.from_numpy(P.b).cuda()) for P in probs], 61, 5,
                 max_iters=4, precision="ff")
    Bt.solve(4)
    xs = [x.cpu().numpy() for x in Bt.x()]
    Bt.close()
    for i in {0, count - 1}:
        ref = O.sgks(probs[i])["x"]
        assert np.linalg.norm(xs[i] - ref) <= 1e-10 * np.linalg.norm(ref)
