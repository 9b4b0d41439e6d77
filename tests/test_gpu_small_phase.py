"""The FP64 cluster kernels (k_small2.cu) at the edges of their plans: sketches with fewer rows than the
cluster has CTAs, basis sizes for which only one exchange buffer fits in shared memory, one and two
Gram-Schmidt passes, refinement.  Iterates against the oracle at the FP64 bar, 1e-10."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads import small_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


# s = 2048 with d_max = 190: one buffer in the QR append; d_max = 393: one buffer in the stacked solve
@pytest.mark.parametrize("s,max_iters,iters,passes,refine", [(9, 3, 3, 2, 0), (13, 8, 5, 2, 1), (17, 10, 6, 1, 0),
                                                             (33, 20, 8, 2, 0), (120, 40, 10, 2, 2), (2048, 187, 8, 2, 1),
                                                             (2048, 187, 8, 1, 0), (400, 390, 8, 2, 0)])
def test_small_phase(G, s, max_iters, iters, passes, refine):
    P = small_problem("deblur2d", nx=32, ny=24, s=s, lam=0.5, precision="fp64", n_refine=refine, iters=iters)
    kw = G.device_inputs(P, "fp64")
    kw["max_iters"] = max_iters
    S = G.Solver(**kw, cgs_passes=passes)
    out = S.solve(iters)
    x = S.x().cpu().numpy()
    S.close()
    assert out["iters_done"] == iters
    ref = O.sgks(P, iters=iters, cgs_passes=passes)["x"]
    assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)
