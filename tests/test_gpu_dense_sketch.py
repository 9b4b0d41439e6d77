"""Dense sketches (k_dense.cu) at the edges of their row groups (2 or 8 rows) and column chunks
(1,024 columns or more): S v for one vector, and the pair S_A A w, S_L L w of an appended column."""
import pytest
import torch

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_18073_gb300 as G
    G.build()
    return G


def solver(G, nx, ny, s, seed=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    m, p = nx * ny, 2 * nx * ny - nx - ny
    SA, SL = (torch.randn(s, h, generator=g, dtype=torch.float64, device="cuda") for h in (m, p))
    b = torch.randn(m, generator=g, dtype=torch.float64, device="cuda")
    psf = torch.rand(3, 3, generator=g, device="cuda")
    S = G.Solver(G.Conv2D(psf, nx, ny), G.Reg("grad2d", nx, ny), b, 0.1, s, 0, max_iters=3, sketch="gaussian",
                 gauss_SA=SA, gauss_SL=SL)
    return S, SA, SL, m, p


# m = nx ny, p = 2 nx ny - nx - ny; s (m + p) below 2^20 takes 2 rows per group, from there on 8
@pytest.mark.parametrize("nx,ny,s", [(7, 5, 9), (32, 32, 12), (33, 31, 31), (41, 25, 33), (64, 16, 340), (91, 90, 43),
                                     (256, 17, 401), (300, 100, 130)])
def test_dense_sketch_edges(G, nx, ny, s):
    S, SA, SL, m, p = solver(G, nx, ny, s)
    L = G._lib
    for which, M in ((L.SGKS_APPLY_SA, SA), (L.SGKS_APPLY_SL, SL)):
        h = M.shape[1]
        v = torch.randn(h, dtype=torch.float64, device="cuda")
        out = torch.full((s,), float("nan"), dtype=torch.float64, device="cuda")
        S.apply(which, v, out)
        # any order of summation: at most h roundings per term, of both results
        assert ((out - M @ v).abs() <= 2 * h * U * (M.abs() @ v.abs())).all()
    # the pair: Q R of the factors the setup built is the sketched basis (CGS2: a few roundings of
    # the column per append on top of the products')
    d, dm = 3, 6
    W = S.buffer(L.SGKS_BUF_W, dm * m).view(-1, m)[:d]
    AW = S.buffer(L.SGKS_BUF_AW, dm * m).view(-1, m)[:d]
    img = W.view(d, ny, nx)
    LW = torch.cat([img.diff(dim=2).reshape(d, -1), img.diff(dim=1).reshape(d, -1)], 1)
    for M, V, bq, br in ((SA, AW, L.SGKS_BUF_QA, L.SGKS_BUF_RA), (SL, LW, L.SGKS_BUF_QL, L.SGKS_BUF_RL)):
        Q = S.buffer(bq, dm * s).view(-1, s)[:d]
        R = S.buffer(br, dm * dm).view(-1, dm)[:d, :d].tril()   # row j: column j of R, written to the diagonal
        got, want = R @ Q, V @ M.T
        bound = 2 * M.shape[1] * U * (V.abs() @ M.abs().T) + 64 * U * want.norm(dim=1, keepdim=True)
        assert ((got - want).abs() <= bound).all()
    S.close()
