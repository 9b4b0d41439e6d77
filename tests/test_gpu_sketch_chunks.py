"""Sparse-sign sketches of the compensated batches by column chunks (k_sketchx.cu): sketch sizes that do not
fill the groups of four rows, chunks that end inside the vectors, one to sixteen entries per column, every
lane layout and every regularizer.  Compared with the oracle at the float-float bar, 1e-10."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads.problem import OperatorDesc, Problem, RegDesc, SketchDesc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


def dense(m, reg, seed):
    rng = np.random.default_rng(seed)
    D = rng.uniform(-1.0, 1.0, (m, reg.n)).astype(np.float32).astype(np.float64) / 16.0
    return OperatorDesc("dense", m, reg.n, dense=D)


REGS = {"fd1": RegDesc("fd1", nx=300), "grad2d": RegDesc("grad2d", nx=17, ny=20),
        "laplace2d": RegDesc("laplace2d", nx=16, ny=16), "spacetime": RegDesc("spacetime", nx=7, ny=9, nt=5)}


# m: one row short of, at and past a chunk's 256 columns, and below one
@pytest.mark.parametrize("reg,m,s,zeta,count", [("fd1", 255, 17, 1, 1), ("fd1", 256, 50, 8, 2), ("grad2d", 257, 61, 16, 3),
                                                ("grad2d", 90, 203, 8, 16), ("laplace2d", 513, 24, 5, 9),
                                                ("spacetime", 300, 35, 8, 1), ("spacetime", 700, 130, 8, 33)])
def test_sketch_chunks(G, reg, m, s, zeta, count):
    L = REGS[reg]
    A = dense(m, L, 1)
    rng = np.random.default_rng(2)
    probs = []
    for i in range(count):
        x = rng.uniform(0.0, 1.0, L.n).astype(np.float32).astype(np.float64)
        b = (A.dense @ x * (1.0 + 0.05 * rng.standard_normal(m))).astype(np.float32).astype(np.float64)
        probs.append(Problem("t", A, L, b, x, 10.0 ** rng.uniform(-1, 0), 4, SketchDesc("sparse_sign", s, zeta, 7)))
    kw = G.device_inputs(probs[0], "ff")
    Bt = G.Batch([dict(A=kw["A"], reg=kw["reg"], lam=P.lam, b=torch.from_numpy(P.b).cuda()) for P in probs], s, 7,
                 max_iters=4, precision="ff", zeta=zeta)
    Bt.solve(4)
    xs = [x.cpu().numpy() for x in Bt.x()]
    Bt.close()
    for P, x in zip(probs, xs):
        ref = O.sgks(P)["x"]
        assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)
