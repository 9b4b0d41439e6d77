"""Memory that the build of the tiled layouts (k_tile_build.cu) takes for a while."""
import ctypes

import numpy as np
import pytest
import torch

from workloads.configs import blockdiag_csr, ct_op

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


class Pool:
    """High-water mark of the device's default memory pool, from which the build takes its temporaries."""
    USED_HIGH = 8   # cudaMemPoolAttrUsedMemHigh

    def __init__(self):
        self.rt = ctypes.CDLL("libcudart.so.13")
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def reset(self):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, self.USED_HIGH, ctypes.byref(v)) == 0

    def high(self):
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolGetAttribute(self.pool, self.USED_HIGH, ctypes.byref(v)) == 0
        return v.value


@pytest.mark.parametrize("form", ["single", "ff"])
def test_temporaries_of_many_frames(G, form):
    """A tile is crossed by its own frame's rays only, so the temporaries stay below 16 bytes per entry (three
    words per segment, at most an entry each, and the frame's bits) however many frames there are."""
    op = ct_op(32, np.arange(8) * 22.5, 46)
    A = blockdiag_csr([op] * 768)
    assert A.val.size >= 1 << 20
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    C = G.CSR(dev(A.row_ptr), dev(A.col), dev(A.val.astype(np.float32)), A.m, A.n).transposed()
    reg = G.Reg("spacetime", 32, 32, 768)
    b = torch.ones(A.m, dtype=torch.float64, device="cuda")
    pool = Pool()
    torch.cuda.synchronize()
    pool.reset()
    S = (G.Solver(C, reg, b, 1.0, 40, 3, max_iters=3) if form == "single" else
         G.Batch([dict(A=C, reg=reg, lam=1.0, b=b)], 40, 3, max_iters=3, precision="ff"))
    high = pool.high()
    S.close()
    assert 0 < high <= 16 * A.val.size
