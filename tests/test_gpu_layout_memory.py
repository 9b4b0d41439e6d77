"""Tiled layouts of a CSR operator (k_tile_build.cu) when device memory is short: they are an option, so a handle
for which the rest fits is created on the row kernels."""
import gc

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


@pytest.fixture(scope="module")
def lines(G):
    """Rays along x on a 512^2 image, 256 pixels each: 30 M entries, 240 MB a layout and as much again for the
    operator, its transpose and the slices of a single FP64 handle."""
    N, m, k = 512, 120000, 256
    g = torch.Generator(device="cuda").manual_seed(1)
    y = torch.randint(0, N, (m, 1), generator=g, device="cuda")
    x0 = torch.randint(0, N - k, (m, 1), generator=g, device="cuda")
    col = (y * N + x0 + torch.arange(k, device="cuda")).to(torch.int32).reshape(-1)
    val = torch.rand(m * k, generator=g, device="cuda") + 0.1
    rp = (torch.arange(m + 1, device="cuda") * k).to(torch.int32)
    A = G.CSR(rp, col, val, m, N * N).transposed()
    return dict(A=A, reg=G.Reg("grad2d", N, N), b=torch.rand(m, generator=g, device="cuda", dtype=torch.float64))


def solve(G, lines, form):
    A, reg, b = lines["A"], lines["reg"], lines["b"]
    if form == "single":
        S = G.Solver(A, reg, b, 1.0, 60, 3, max_iters=5)
    else:
        S = G.Batch([dict(A=A, reg=reg, lam=1.0, b=b), dict(A=A, reg=reg, lam=2.0, b=b)], 60, 3, max_iters=5, precision=form)
    S.solve(5)
    x = S.x()
    S.close()
    return [v.clone() for v in x] if isinstance(x, list) else [x.clone()]


# free memory at the handle's creation, MB.  The handles need 380 (single), 120 (fp64) and 190 (ff) without layouts
# and about 600 more for both of them and their building, so that either of them, or both, have no room.
@pytest.mark.parametrize("form,free", [("single", 700), ("single", 900), ("fp64", 500), ("fp64", 700), ("ff", 600),
                                       ("ff", 800)])
def test_handle_without_room_for_layouts(G, lines, form, free):
    ref = solve(G, lines, form)
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (free << 20), dtype=torch.uint8, device="cuda")
    try:
        xs = solve(G, lines, form)
    finally:
        del hold
        torch.cuda.empty_cache()
    for x, r in zip(xs, ref):
        assert torch.linalg.norm(x - r) <= 1e-10 * torch.linalg.norm(r)


def test_reverse_sweep_without_room_beside_the_layouts(G, lines):
    """The sweep's workspace (17 MB and more) is allocated at its first call; the layouts then make room."""
    kw = dict(max_iters=5, record=True)
    xbar = torch.rand(lines["A"].n, device="cuda", dtype=torch.float64)
    S = G.Solver(lines["A"], lines["reg"], lines["b"], 1.0, 60, 3, **kw)
    S.solve(5)
    ref, lref = S.backward(xbar)
    S.close()
    S = G.Solver(lines["A"], lines["reg"], lines["b"], 1.0, 60, 3, **kw)
    S.solve(5)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    mine = torch.empty(16 << 20, dtype=torch.uint8, device="cuda")
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (12 << 20), dtype=torch.uint8, device="cuda")
    del mine     # stays with torch's allocator, for the result
    try:
        bb, lb = S.backward(xbar)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.linalg.norm(bb - ref) <= 1e-10 * torch.linalg.norm(ref) and abs(lb - lref) <= 1e-10 * abs(lref)
    S.reset(lines["b"])
    S.solve(5)   # on the row kernels now
    b2, _ = S.backward(xbar)
    S.close()
    assert torch.linalg.norm(b2 - ref) <= 1e-10 * torch.linalg.norm(ref)
