"""What the tuner has measured for one kind of passes is not taken for another kind (SGKS_FLAG_AUTOTUNE)."""
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


@pytest.mark.parametrize("prec,count,N", [("ff", 16, 45), ("fp64", 4, 192)])
@pytest.mark.parametrize("first", [True, False])
def test_tiled_and_row_passes_are_tuned_apart(G, prec, count, N, first):
    A = ct_op(N, np.arange(100) * 1.8, int(1.43 * N) + int(first))   # a shape of its own per order
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    C = G.CSR(dev(A.row_ptr), dev(A.col), dev(A.val.astype(np.float32)), A.m, A.n).transposed()
    b = torch.ones(A.m, dtype=torch.float64, device="cuda")
    said = {}
    for tiles in (first, not first, first):
        Bt = G.Batch([dict(A=C, reg=G.Reg("grad2d", N, N), lam=2.0, b=b)] * count, 60, 3, max_iters=5, precision=prec,
                     tiles=tiles, autotune=True)
        said.setdefault(tiles, []).append(Bt.config())
        Bt.close()
    assert said[first][0] != "cached" and said[first][1] == "cached"
    assert said[not first][0] != "cached"


def test_shapes_are_tuned_apart(G):
    """The same numbers of rows, unknowns and entries on images of different sides (their p differs too, unless the
    sides are only swapped)."""
    m, nx, ny = 640, 48, 32
    n = nx * ny
    col = (torch.arange(m * 8, device="cuda") * 37 % n).to(torch.int32).reshape(m, 8).sort(dim=1).values.reshape(-1)
    C = G.CSR((torch.arange(m + 1, device="cuda") * 8).to(torch.int32), col, torch.ones(m * 8, device="cuda"), m, n).transposed()
    b = torch.ones(m, dtype=torch.float64, device="cuda")
    for sides in ((nx, ny), (ny, nx)):
        Bt = G.Batch([dict(A=C, reg=G.Reg("grad2d", *sides), lam=2.0, b=b)], 60, 3, max_iters=5, precision="ff", autotune=True)
        assert Bt.config() != "cached"
        Bt.close()
