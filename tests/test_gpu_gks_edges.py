"""GKS appends (k_gks.cu) at the edges of their tiles of 256 rows, with odd and even numbers of columns, and
with more columns than the CTA has warps: iterates against the oracle's gks() at the FP64 bar, 1e-10."""
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


@pytest.mark.parametrize("nx,ny,iters", [(5, 51, 3), (16, 16, 6), (257, 2, 9), (23, 45, 24)])
def test_gks_edges(G, nx, ny, iters):
    P = small_problem("deblur2d", nx=nx, ny=ny, precision="fp64", n_refine=0, iters=iters, lam=0.1)
    S = G.Solver(**G.device_inputs(P, "fp64"), method="gks")
    S.solve(iters)
    x = S.x().cpu().numpy()
    S.close()
    ref = O.gks(P)["x"]
    assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)
