"""Range of the reverse sweep on an operator that takes the FP64 tiled passes (k_tiles64.cu, from 2^20 entries on):
the derivative is linear in the cotangent, whose scale is the caller's."""
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


def setup(G, refine, scale_A=1.0, scale_b=1.0):
    A = ct_op(97, np.arange(100) * 1.8, 139)
    assert A.val.size >= 1 << 20
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    C = G.CSR(dev(A.row_ptr), dev(A.col), dev(A.val.astype(np.float32)) * scale_A, A.m, A.n).transposed()
    rng = np.random.default_rng(5)
    b = dev(rng.uniform(0.5, 1.5, A.m)) * scale_b
    xbar = dev(rng.standard_normal(A.n))
    S = G.Solver(C, G.Reg("grad2d", 97, 97), b, 2.0 * scale_A**2, 60, 3, max_iters=6, n_refine=refine, record=True)
    S.solve(6)
    return S, xbar


@pytest.mark.parametrize("refine", [0, 1])
def test_cotangents_of_any_scale(G, refine):
    """Powers of two, so that every rounding is the same: bit for bit."""
    S, xbar = setup(G, refine)
    bb, lb = S.backward(xbar)
    for k in (-900, -640, -560, 480, 620, 900):
        b2, l2 = S.backward(xbar * 2.0**k)
        assert torch.equal(b2, bb * 2.0**k)
        assert l2 == lb * 2.0**k
    S.close()


def test_zero_and_infinite_cotangents(G):
    S, xbar = setup(G, 0)
    bb, lb = S.backward(torch.zeros_like(xbar))
    assert lb == 0.0 and not bb.any()
    xbar[17] = float("inf")
    bb, lb = S.backward(xbar)
    assert not torch.isfinite(bb).all()
    S.close()


def test_large_operators_and_data(G):
    """(A^T A)^2 A^T b at the end of the sweep, here of size 2^670, goes through 2^560.  lambda goes with the square of
    A's scale k, so that the solution is that of the plain problem times c / k, c the scale of b."""
    S, xbar = setup(G, 0)
    bb, lb = S.backward(xbar)
    S.close()
    k, c = 2.0**110, 2.0**120
    S, xbar = setup(G, 0, k, c)
    b2, l2 = S.backward(xbar)
    S.close()
    assert torch.linalg.norm(b2 * k - bb) <= 1e-12 * torch.linalg.norm(bb)
    assert abs(l2 / c * k * k * k - lb) <= 1e-12 * abs(lb)
