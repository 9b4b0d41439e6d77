"""Tiled passes of the compensated batches (k_tiles.cu, k_tile_build.cu) where they can go wrong: images that
end inside a tile, several stages of rows per tile, every lane layout (1, 2, 4, 8, 16 instances per CTA), rows
with unsorted entries, empty rows and columns, a row through every pixel, and operators whose
rows share too little of a tile for the transposed pass to be tiled.  Every instance is compared with the
oracle on its own problem at the bar of its form: 1e-10 (float-float), 1e-4 (FP32)."""
import numpy as np
import pytest
import torch

import oracle as O
from workloads.configs import blockdiag_csr, ct_op
from workloads.problem import OperatorDesc, Problem, RegDesc, SketchDesc

pytestmark = pytest.mark.gpu
BAR = {"ff": 1e-10, "fp32": 1e-4}


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


def rays(N, views, frames=1):
    ops = [ct_op(N, np.arange(views) * (180.0 / views) + 3.0 * t, int(1.42 * N) + 1) for t in range(frames)]
    A = ops[0] if frames == 1 else blockdiag_csr(ops)
    return A, RegDesc("spacetime", nx=N, ny=N, nt=frames) if frames > 1 else RegDesc("grad2d", nx=N, ny=N)


def scattered(nx, ny, m, per_row, seed=0):
    """Random entries in random order: row 0 empty, row 2 through every pixel, the last pixel in no row
    but that one (an entry twice is refused by the library)."""
    rng = np.random.default_rng(seed)
    n = nx * ny
    cols = [rng.permutation(n - 1)[:per_row] for _ in range(m)]
    cols[0] = cols[0][:0]
    cols[2] = rng.permutation(n)
    rp = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32)
    val = rng.uniform(0.1, 1.0, rp[-1]).astype(np.float32)
    A = OperatorDesc("csr", m, n, row_ptr=rp, col=np.concatenate(cols).astype(np.int32), val=val, nx=nx, ny=ny)
    return A, RegDesc("laplace2d", nx=nx, ny=ny)


CASES = {
    "rays37": lambda: rays(37, 40),              # 16 x 8 tiles: 760 rows of a tile, two stages of 512
    "rays32_many": lambda: rays(32, 250),        # 16 x 16 tiles: about 6,000 rows of a tile
    "frames": lambda: rays(19, 30, frames=3),
    "scattered_wide": lambda: scattered(45, 21, 400, 60),
    "scattered_thin": lambda: scattered(50, 33, 900, 3),
}


@pytest.mark.parametrize("prec", ["ff", "fp32"])
@pytest.mark.parametrize("name,count", [("rays37", 1), ("rays37", 3), ("rays37", 21), ("rays32_many", 1),
                                        ("rays32_many", 12), ("frames", 2), ("frames", 16), ("scattered_wide", 1),
                                        ("scattered_wide", 6), ("scattered_wide", 16), ("scattered_thin", 9)])
def test_tiled_passes(G, name, count, prec):
    A, L = CASES[name]()
    rng = np.random.default_rng(count)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    probs = []
    for i in range(count):
        x = f32(rng.uniform(0.0, 1.0, A.n))
        b = np.zeros(A.m)
        np.add.at(b, np.repeat(np.arange(A.m), np.diff(A.row_ptr)), A.val.astype(np.float64) * x[A.col])
        b = f32(b * (1.0 + 0.02 * rng.standard_normal(A.m)))
        probs.append(Problem("t", A, L, b, x, 10.0 ** rng.uniform(-1, 1), 5, SketchDesc("sparse_sign", 60, 8, 3),
                             precision=prec))
    kw = G.device_inputs(probs[0], prec)
    dt = G.io_dtype(prec)
    Bt = G.Batch([dict(A=kw["A"], reg=kw["reg"], lam=P.lam, b=torch.from_numpy(P.b).to("cuda", dt)) for P in probs],
                 60, 3, max_iters=5, precision=prec)
    Bt.solve(5)
    xs = [x.double().cpu().numpy() for x in Bt.x()]
    Bt.close()
    for P, x in zip(probs, xs):
        ref = O.sgks(P)["x"]
        assert np.linalg.norm(x - ref) <= BAR[prec] * np.linalg.norm(ref)


def test_columns_outside_the_image_are_refused(G):
    A, L = rays(16, 6)
    A.col = A.col.copy()
    P = Problem("t", A, L, np.ones(A.m), np.ones(A.n), 1.0, 3, SketchDesc("sparse_sign", 40, 8, 0))
    kw = G.device_inputs(P, "ff")          # builds A^T from the valid operator
    kw["A"].col[5] = A.n
    with pytest.raises(Exception):
        G.Batch([dict(A=kw["A"], reg=kw["reg"], lam=1.0, b=kw["b"])], 40, 0, max_iters=3, precision="ff")
