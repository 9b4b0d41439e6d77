"""The limit on a kernel's shared memory belongs to the process, not to a handle: handles of different sizes, one
after the other or in several host threads, do not lower it for each other."""
import threading

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


def blur(G, nx, ny, count, max_iters, precision="ff", refine=0, s=64):
    psf = torch.full((3, 3), 1.0 / 9.0, device="cuda")
    A, reg = G.Conv2D(psf, nx, ny), G.Reg("grad2d", nx, ny)
    g = torch.Generator(device="cuda").manual_seed(nx)
    bs = [torch.rand(nx * ny, generator=g, device="cuda", dtype=torch.float64) for _ in range(count)]
    return G.Batch([dict(A=A, reg=reg, lam=0.1, b=b) for b in bs], s, 1, max_iters=max_iters, precision=precision,
                   n_refine=refine), bs


def test_refinement_of_a_long_basis_beside_a_short_one(G):
    """k_refine_solve2 takes 16 bytes per column of the basis."""
    long, _ = blur(G, 24, 20, 1, 300, "fp64", 1, s=400)
    short, _ = blur(G, 24, 20, 1, 2, "fp64", 1)
    long.solve(4)
    short.solve(2)
    assert all(torch.isfinite(x).all() for x in long.x() + short.x())
    long.close()
    short.close()


def test_two_threads_with_different_chunks(G):
    """64 instances of 96 x 96 take sketch chunks of 384 columns, of 200 x 160 ones of 768 (k_sketchx.cu)."""
    pairs = [blur(G, 96, 96, 64, 4), blur(G, 200, 160, 64, 4)]
    errors = []

    def work(Bt, bs):
        try:
            for _ in range(1500):
                Bt.reset(bs)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    torch.cuda.synchronize()
    ts = [threading.Thread(target=work, args=p) for p in pairs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for Bt, _ in pairs:
        Bt.close()
    assert not errors
