"""FP64 tiled passes (k_tiles64.cu, from 2^20 entries on): images that end inside a tile, several frames, every
lane layout, operator values down to FP32 subnormals and of both signs, infinite ones, a full basis.  Compared
with the oracle at the FP64 bar, 1e-10, and with the row kernels."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads.configs import blockdiag_csr, ct_op
from workloads.problem import Problem, RegDesc, SketchDesc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


def operator(name):
    if name == "frames":
        A = blockdiag_csr([ct_op(35, np.arange(100) * 1.8 + t, 51) for t in range(8)])
        L = RegDesc("spacetime", nx=35, ny=35, nt=8)
    else:
        A = ct_op(97, np.arange(100) * 1.8, 139)
        L = RegDesc("grad2d" if name == "grad" else "laplace2d", nx=97, ny=97)
    rng = np.random.default_rng(4)
    k = rng.integers(0, A.val.size, 3000)
    A.val[k[:1000]] *= -1.0
    A.val[k[1000:2000]] = 0.0
    A.val[k[2000:]] = np.float32(1e-41)      # subnormal
    assert A.val.size >= 1 << 20
    return A, L


def problems(name, count):
    A, L = operator(name)
    M = (A.row_ptr, A.col, A.val.astype(np.float64))
    rng = np.random.default_rng(count)
    out = []
    for i in range(count):
        x = rng.uniform(0.0, 1.0, A.n).astype(np.float32).astype(np.float64)
        b = np.add.reduceat(np.append(M[2] * x[M[1]], 0.0), M[0][:-1]) * (np.diff(M[0]) > 0)
        b = (b * (1.0 + 0.02 * rng.standard_normal(A.m))).astype(np.float32).astype(np.float64)
        out.append(Problem("t", A, L, b, x, 10.0 ** rng.uniform(0, 1), 5, SketchDesc("sparse_sign", 60, 8, 3)))
    return out


@pytest.mark.parametrize("name", ["grad", "laplace", "frames"])
def test_single(G, name):
    P = problems(name, 1)[0]
    kw = G.device_inputs(P, "fp64")
    S = G.Solver(**kw)
    S.solve(5)
    x = S.x().cpu().numpy()
    with pytest.raises(Exception):
        S.step()                              # the basis is full
    S.close()
    ref = O.sgks(P)["x"]
    assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)
    S = G.Solver(**{**kw, "n_refine": 0}, method="gks")
    S.solve(5)
    x = S.x().cpu().numpy()
    S.close()
    ref = O.gks(P)["x"]
    assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("name,count,refine", [("grad", 1, 0), ("grad", 7, 1), ("laplace", 24, 0), ("frames", 16, 1)])
def test_batch(G, name, count, refine):
    probs = problems(name, count)
    kw = G.device_inputs(probs[0], "fp64")
    insts = [dict(A=kw["A"], reg=kw["reg"], lam=P.lam, b=torch.from_numpy(P.b).cuda()) for P in probs]
    xs = []
    for tiles in (True, False):
        Bt = G.Batch(insts, 60, 3, max_iters=5, precision="fp64", tiles=tiles, n_refine=refine)
        Bt.solve(5)
        xs.append([x.cpu().numpy() for x in Bt.x()])
        Bt.close()
    for i, P in enumerate(probs):
        ref = O.sgks(P, n_refine=refine)["x"] if i in (0, count - 1) else xs[1][i]
        for x in (xs[0][i], xs[1][i]):
            assert np.linalg.norm(x - ref) <= 1e-10 * np.linalg.norm(ref)


def test_infinite_value_is_reported(G):
    P = problems("grad", 1)[0]
    P.A.val[12345] = np.inf
    with pytest.raises(Exception):
        S = G.Solver(**G.device_inputs(P, "fp64"))
        S.solve(5)
