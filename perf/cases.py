"""Performance cases of the sGKS library: what a program that uses it has it do.

A case is one whole solve (setup and a fixed number of iterations) through ``Solver``, ``Batch`` or
``solve_differentiable`` on a problem of one of the operator families that the library serves:
dense 1-D deconvolution, image deblurring (2-D convolution), parallel-beam CT and travel-time
tomography (CSR), and dynamic CT (block-diagonal CSR with a space-time regularizer).

``listed()`` holds the fixed cases, ``draw(rng)`` gives others of the same ranges, ``prepare`` builds
the inputs and the handle that a program keeps between solves, ``run`` is one solve of a new right-hand
side on that handle, ``work`` counts what the solve cannot do without and ``exact`` is the same
algorithm in plain torch, in float64 throughout.

Iteration counts end where the iterates of the never re-orthogonalised basis still determine a float64
result to far more digits than a comparison needs.
"""
import math

import numpy as np
import torch

import paper_2606_18073_gb300 as G

DEV = "cuda"
F64 = torch.float64
ELL = 3      # dimension of the initial Krylov space
ZETA = 8     # nonzeros per column of the sparse-sign sketch


# ------------------------------------------------------------------------------------- cases

def _case(name, family, api, n, iters, s, precision="fp64", **kw):
    c = dict(name=name, family=family, api=api, n=n, ny=n, iters=iters, s=s, precision=precision, refine=0,
             batch=1, sketch="sparse_sign", method="sgks", views=0, bins=0, frames=1, sides=0)
    c.update(kw)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # the smallest problem in use: 1-D deconvolution with a Gaussian sketch; launches and the
        # small FP64 factorisations are all there is
        _case("deconv_fp64", "deconv", "solver", 256, 30, 120, sketch="gaussian"),
        # one image deblurred in plain FP64
        _case("deblur_fp64", "deblur", "solver", 256, 30, 400),
        # the same in the FP32 form with two refinement steps per iteration
        _case("deblur_fp32_refined", "deblur", "solver", 256, 25, 400, precision="fp32", refine=2),
        # deblurring with the trigonometric sketch (SRTT) that the paper itself uses
        _case("deblur_srtt", "deblur", "solver", 256, 25, 400, sketch="srtt"),
        # Algorithm 1 (GKS, orthonormal basis and full-size QR) on an image of odd shape
        _case("deblur_gks", "deblur", "solver", 201, 30, 0, ny=157, method="gks"),
        # one CT slice in plain FP64: every pass reads the operator once for a single vector
        _case("ct_fp64", "ct", "solver", 512, 40, 600, views=180, bins=725),
        # one CT slice of odd size as a batch of one in the float-float form
        _case("ct_one_ff", "ct", "batch", 301, 30, 300, precision="ff", views=123, bins=427),
        # the many-slices workload: 64 right-hand sides and regularization parameters share one scanner
        _case("ct_batch64_ff", "ct", "batch", 512, 30, 600, precision="ff", batch=64, views=180, bins=725),
        # a ragged number of slices (groups of 8, 2 and 1) of an odd-sized scanner, FP32 form
        _case("ct_batch11_fp32", "ct", "batch", 243, 20, 300, precision="fp32", batch=11, views=97, bins=345),
        # travel-time tomography, several data sets at once in plain FP64
        _case("seismic_batch16_fp64", "seismic", "batch", 256, 30, 400, batch=16, sides=64),
        # learning: the solve and its derivative by the data and the regularization parameter
        _case("seismic_train", "seismic", "train", 256, 20, 400, sides=64),
        # dynamic CT series of different lengths, FP32 form with three refinement steps
        _case("dynct_batch_fp32_refined", "dynct", "batch", 128, 30, 800, precision="fp32", refine=3, batch=6,
              views=30, bins=185, frames=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a family in one of the forms in which the listed cases have it, at another size."""
    kind = rng.choice(["deconv", "deblur", "deblur_fp32", "srtt", "gks", "ct", "ct_one", "ct_batch", "ct_batch",
                       "seismic_batch", "train", "dynct"])
    iters = rng.randint(12, 30)
    s = rng.randint(3, 8) * 50 + rng.randint(0, 99)
    if kind == "deconv":
        n = _log(rng, 128, 640)
        it = rng.randint(10, 30)
        return _case(None, "deconv", "solver", n, it, rng.randint(3 * (it + ELL), n - 1), sketch="gaussian")
    if kind in ("deblur", "deblur_fp32", "srtt", "gks"):
        n = _log(rng, 64, 384)
        ny = _log(rng, max(64, n // 2), min(384, 2 * n))
        if kind == "gks":
            return _case(None, "deblur", "solver", n, iters, 0, ny=ny, method="gks")
        if kind == "srtt":
            n, ny = min(n, 256), min(ny, 256)
            return _case(None, "deblur", "solver", n, min(iters, 16), s + 100, ny=ny, sketch="srtt")
        if kind == "deblur_fp32":
            return _case(None, "deblur", "solver", n, min(iters, 25), s, ny=ny, precision="fp32",
                         refine=rng.choice([0, 1, 2]))
        return _case(None, "deblur", "solver", n, iters, s, ny=ny)
    if kind in ("ct", "ct_one", "ct_batch"):
        n = _log(rng, 64, 420)
        views, bins = rng.randint(48, 140), int(1.4143 * n) + rng.randint(0, 3)
        if kind == "ct":
            prec = rng.choice(["fp64", "fp64", "fp32"])
            return _case(None, "ct", "solver", n, min(iters, 20) if prec == "fp32" else iters, s, views=views,
                         bins=bins, precision=prec)
        B = 1 if kind == "ct_one" else _log(rng, 2, 64)
        prec = rng.choice(["ff", "ff", "fp32"])
        return _case(None, "ct", "batch", n, min(iters, 20 if prec == "fp32" else 26), s, views=views, bins=bins,
                     batch=B, precision=prec)
    if kind == "seismic_batch":
        n = _log(rng, 48, 256)
        return _case(None, "seismic", "batch", n, min(iters, 26), s, batch=_log(rng, 2, 24),
                     sides=rng.randint(24, 64), precision=rng.choice(["fp64", "ff", "fp32"]))
    if kind == "train":
        n = _log(rng, 48, 256)
        return _case(None, "seismic", "train", n, rng.randint(8, 20), s, sides=rng.randint(24, 64))
    n = _log(rng, 40, 128)
    return _case(None, "dynct", "batch", n, min(iters, 26), s, precision="fp32", refine=rng.randint(1, 3),
                 batch=rng.randint(2, 6), views=rng.randint(12, 30), bins=int(1.4143 * n) + rng.randint(1, 4),
                 frames=rng.randint(4, 16))


# ------------------------------------------------------------------------------- problem data

def _rng(seed, stream):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, int(stream)])


def _f32(x):
    return x.to(torch.float32).to(F64)


def _trace(p0, p1, N):
    """Intersection lengths of the segments p0 -> p1 with the unit pixels of [0, N]^2 (Siddon):
    per segment count, then pixel index and length of every crossing, segment by segment."""
    counts, cols, vals = [], [], []
    step = max(1, (1 << 25) // (2 * N + 4))
    k = torch.arange(N + 1, dtype=F64, device=DEV)
    for a in range(0, p0.shape[0], step):
        q0, d = p0[a:a + step], p1[a:a + step] - p0[a:a + step]
        length = torch.hypot(d[:, 0], d[:, 1])
        flat = d.abs() < 1e-12
        t = (k[None, None, :] - q0[:, :, None]) / torch.where(flat, torch.ones_like(d), d)[:, :, None]
        lo, hi = torch.minimum(t[..., 0], t[..., N]), torch.maximum(t[..., 0], t[..., N])
        inside = (q0 >= 0) & (q0 <= N)
        lo = torch.where(flat, torch.where(inside, -torch.inf, torch.inf), lo).amax(1).clamp_min(0.0)
        hi = torch.where(flat, torch.where(inside, torch.inf, -torch.inf), hi).amin(1).clamp_max(1.0)
        hi = torch.maximum(hi, lo.clamp_max(1.0))
        lo = torch.minimum(lo, hi)
        t = torch.where(flat[:, :, None], lo[:, None, None], t).reshape(q0.shape[0], -1)
        t = torch.cat([t, lo[:, None], hi[:, None]], 1)
        t = torch.minimum(torch.maximum(t, lo[:, None]), hi[:, None]).sort(1).values
        seg = (t[:, 1:] - t[:, :-1]) * length[:, None]
        mid = 0.5 * (t[:, 1:] + t[:, :-1])
        ix = (q0[:, 0:1] + mid * d[:, 0:1]).floor().long()
        iy = (q0[:, 1:2] + mid * d[:, 1:2]).floor().long()
        ok = (seg > 1e-6) & (ix >= 0) & (ix < N) & (iy >= 0) & (iy < N)
        row = torch.arange(q0.shape[0], device=DEV)[:, None].expand_as(ok)[ok]
        key, order = (row * (N * N) + (iy * N + ix)[ok]).sort()
        counts.append(torch.bincount(row, minlength=q0.shape[0]))
        cols.append((key % (N * N)).to(torch.int32))
        vals.append(seg[ok][order].to(torch.float32))
    return torch.cat(counts), torch.cat(cols), torch.cat(vals)


def _parallel(N, angles, bins):
    """Rays of a parallel beam: angle-major, detector bins of one pixel around the image centre."""
    th = torch.as_tensor(angles, dtype=F64, device=DEV)
    nrm = torch.stack([th.cos(), th.sin()], 1)
    along = torch.stack([-th.sin(), th.cos()], 1)
    u = torch.arange(bins, dtype=F64, device=DEV) - (bins - 1) / 2.0
    mid = N / 2.0 + u[None, :, None] * nrm[:, None, :]
    half = (0.75 * N + 2.0) * along[:, None, :]
    return (mid - half).reshape(-1, 2), (mid + half).reshape(-1, 2)


def _csr(case, frames):
    """(row_ptr, col, val, m, n) of the case's ray operator with `frames` frames."""
    N = case["n"]
    if case["family"] == "seismic":
        k = case["sides"]
        y = (torch.arange(k, dtype=F64, device=DEV) + 0.5) * (N / k)
        src = torch.stack([torch.zeros_like(y), y], 1)
        rec = torch.cat([torch.stack([torch.full_like(y, N), y], 1), torch.stack([y, torch.full_like(y, N)], 1)])
        p0 = src[:, None, :].expand(k, 2 * k, 2).reshape(-1, 2)
        p1 = rec[None, :, :].expand(k, 2 * k, 2).reshape(-1, 2)
    elif case["family"] == "dynct":
        a = [((6.0 * t + 0.2 * j) % 180.0) * math.pi / 180.0 for t in range(frames) for j in range(case["views"])]
        p0, p1 = _parallel(N, a, case["bins"])
    else:
        p0, p1 = _parallel(N, [j * math.pi / case["views"] for j in range(case["views"])], case["bins"])
    counts, col, val = _trace(p0, p1, N)
    m = counts.numel()
    rp = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=rp[1:])
    if frames > 1:
        frame = torch.arange(m, device=DEV) // (m // frames)
        col = col + (torch.repeat_interleave(frame, counts) * (N * N)).to(torch.int32)
    return rp.to(torch.int32), col, val, m, N * N * frames


def _psf():
    r = torch.arange(9, dtype=F64, device=DEV) - 4
    h = torch.exp(-(r[:, None] ** 2 + r[None, :] ** 2) / 8.0)
    return (h / h.sum()).to(torch.float32)


def _blur_matrix(n):
    i = torch.arange(n, dtype=F64, device=DEV)
    D = (i[:, None] - i[None, :]).abs()
    A = torch.where(D <= 12, torch.exp(-D ** 2 / 18.0), torch.zeros_like(D))
    return (A / A.sum(1, keepdim=True)).to(torch.float32)


def _conv(psf, img, adjoint=False):
    """2-D convolution (or its adjoint) of (..., ny, nx) with zero boundary, tap by tap."""
    kh, kw = psf.shape
    ny, nx = img.shape[-2:]
    pad = torch.nn.functional.pad(img, (kw // 2, kw // 2, kh // 2, kh // 2))
    out = torch.zeros_like(img)
    for a in range(kh):
        for c in range(kw):
            da, dc = (a, c) if adjoint else (kh - 1 - a, kw - 1 - c)
            out = out + psf[a, c] * pad[..., da:da + ny, dc:dc + nx]
    return out


def _ellipses(N, frames, rng, count):
    yy, xx = torch.meshgrid(*(2 * [torch.arange(N, dtype=F64, device=DEV) + 0.5]), indexing="ij")
    vol = torch.zeros(frames, N, N, dtype=F64, device=DEV)
    for _ in range(count):
        cx, cy = rng.uniform(0.3 * N, 0.7 * N, 2)
        a, b = rng.uniform(0.04 * N, 0.22 * N, 2)
        ang, way, speed, dens = rng.uniform(0, math.pi), rng.uniform(0, 2 * math.pi), rng.choice([1.0, 2.0]), rng.uniform(0.1, 1)
        for t in range(frames):
            dx, dy = xx - (cx + t * speed * math.cos(way)), yy - (cy + t * speed * math.sin(way))
            u, v = (math.cos(ang) * dx + math.sin(ang) * dy) / a, (math.cos(ang) * dy - math.sin(ang) * dx) / b
            vol[t] += dens * ((u * u + v * v) <= 1.0)
    return _f32(vol.reshape(-1))


def _phantom(case, frames, seed):
    rng, n, ny = _rng(seed, 0), case["n"], case["ny"]
    if case["family"] == "deconv":   # piecewise constant
        cuts = np.sort(rng.choice(np.arange(1, n), 4, replace=False))
        return _f32(torch.from_numpy(rng.uniform(0, 1, 5)[np.searchsorted(cuts, np.arange(n), "right")]).to(DEV))
    if case["family"] == "deblur":   # rectangles, later ones on top
        img = torch.zeros(ny, n, dtype=F64, device=DEV)
        for _ in range(20):
            x, y = np.sort(rng.integers(0, n + 1, 2)), np.sort(rng.integers(0, ny + 1, 2))
            img[y[0]:max(y[1], y[0] + 1), x[0]:max(x[1], x[0] + 1)] = rng.uniform(0, 1)
        return _f32(img.reshape(-1))
    if case["family"] == "seismic":  # a smooth random slowness field around 1
        w = torch.from_numpy(rng.standard_normal((n, n))).to(DEV)
        k = torch.fft.fftfreq(n, dtype=F64, device=DEV)
        f = torch.fft.ifft2(torch.fft.fft2(w) * torch.exp(-4.0 * n * (k[:, None] ** 2 + k[None, :] ** 2))).real
        return _f32((1.0 + 0.1 * (f - f.mean()) / f.std()).reshape(-1))
    return _ellipses(n, frames, rng, 4 if frames > 1 else 10)


def _noisy(bt, level, seed, stream):
    g = torch.Generator(device=DEV).manual_seed((int(seed) * 1009 + stream) & 0x7FFFFFFF)
    e = torch.randn(bt.numel(), generator=g, dtype=F64, device=DEV)
    return _f32(bt + e * (level * bt.norm() / e.norm()))


NOISE = {"deconv": 0.01, "deblur": 0.01, "ct": 0.02, "seismic": 0.01, "dynct": 0.01}
LAM = {"deconv": 1e-2, "deblur": 5e-3, "ct": 1e-2, "seismic": 2.7, "dynct": 27.0}
REG = {"deconv": "fd1", "deblur": "grad2d", "ct": "grad2d", "seismic": "laplace2d", "dynct": "spacetime"}


class _Problem:
    """One operator with the right-hand sides that share it: A (as stored), b [k][m], lam [k]."""

    def __init__(self, case, seed, frames, which):
        fam, n, ny = case["family"], case["n"], case["ny"]
        self.family, self.frames, self.nx = fam, frames, n
        self.ny = 1 if fam == "deconv" else ny if fam == "deblur" else n
        x = _phantom(case, frames, seed)
        self.n, self.x_true = x.numel(), x
        if fam == "deconv":
            self.dense = _blur_matrix(n)
            bt = self.dense.to(F64) @ x
        elif fam == "deblur":
            self.psf = _psf()
            bt = _conv(self.psf.to(F64), x.view(ny, n)).reshape(-1)
        else:
            rp, col, val, m, _ = self.csr = _csr(case, frames)
            bt = torch.segment_reduce(val.to(F64) * x[col.long()], "sum", offsets=rp.long(), axis=0, initial=0.0)
        self.m = bt.numel()
        self.b = [_noisy(bt, NOISE[fam], seed, i) for i in which]
        k = len(which)
        # one regularization parameter for a single data set, a range of them for a batch
        self.lam = [LAM[fam]] if k == 1 else [LAM[fam] * 10.0 ** (3.0 * i / (k - 1) - 1.5) for i in range(k)]

    def op(self):
        if self.family == "deconv":
            return G.Dense(self.dense)
        if self.family == "deblur":
            return G.Conv2D(self.psf, self.nx, self.ny)
        rp, col, val, m, n = self.csr
        return G.CSR(rp, col, val, m, n).transposed()

    def reg(self):
        return G.Reg(REG[self.family], self.nx, self.ny, self.frames)

    def p(self):
        nx, ny, nt = self.nx, self.ny, self.frames
        if self.family == "deconv":
            return nx - 1
        if self.family == "seismic":
            return nx * ny
        return nt * (ny * (nx - 1) + (ny - 1) * nx) + (nt - 1) * nx * ny


def _problems(case, seed):
    """The operators of a case, each with its right-hand sides: dynamic CT batches hold series of
    different lengths (half of them half as long), the other cases one operator."""
    B, F = case["batch"], case["frames"]
    if case["family"] == "dynct" and B > 1:
        return [_Problem(case, seed, F, list(range(0, B, 2))), _Problem(case, seed, max(2, F // 2), list(range(1, B, 2)))]
    return [_Problem(case, seed, F, list(range(B)))]


def _sketch_inputs(case, seed, m, p):
    rng, s = _rng(seed, 7), case["s"]
    if case["sketch"] == "gaussian":
        g = torch.Generator(device=DEV).manual_seed((int(seed) * 1013 + 5) & 0x7FFFFFFF)
        return [torch.randn(s, h, generator=g, dtype=F64, device=DEV) / math.sqrt(s) for h in (m, p)]
    got = []
    for h in (m, p):
        got += [torch.from_numpy(rng.choice(np.array([-1, 1], np.int8), h)).to(DEV),
                torch.from_numpy(np.sort(rng.choice(h, s, replace=False)).astype(np.int32)).to(DEV)]
    return got


# ------------------------------------------------------------------------------ prepare / run

def prepare(case, seed):
    prec = case["precision"]
    dt = G.io_dtype(prec)
    probs = _problems(case, seed)
    sk = int(seed) & 0x7FFFFFFF
    st = dict(case=case)
    if case["api"] == "batch":
        insts = []
        for P in probs:
            A, reg = P.op(), P.reg()
            insts += [dict(A=A, reg=reg, b=b.to(dt), lam=lam) for b, lam in zip(P.b, P.lam)]
        st["b"] = [i["b"] for i in insts]
        st["solver"] = G.Batch(insts, case["s"], sk, max_iters=case["iters"], n_refine=case["refine"], precision=prec,
                               zeta=ZETA)
        st["x"] = [torch.empty(len(P.b), P.n, dtype=dt, device=DEV) for P in probs]
        st["rows"] = [row for x in st["x"] for row in x]
        return st
    P = probs[0]
    kw = dict(max_iters=case["iters"], n_refine=case["refine"], precision=prec, zeta=ZETA, sketch=case["sketch"],
              method=case["method"], record=case["api"] == "train")
    s = case["s"] or 2 * (case["iters"] + ELL)
    if case["sketch"] == "gaussian":
        kw["gauss_SA"], kw["gauss_SL"] = _sketch_inputs(case, seed, P.m, P.p())
    elif case["sketch"] == "srtt":
        kw["srtt"] = tuple(_sketch_inputs(case, seed, P.m, P.p()))
    st["b"] = P.b[0].to(dt)
    st["solver"] = G.Solver(P.op(), P.reg(), st["b"], P.lam[0], s, sk, **kw)
    st["x"] = torch.empty(P.n, dtype=dt, device=DEV)
    if case["api"] == "train":
        st["x_true"] = P.x_true
        st["lam"] = torch.tensor(P.lam[0], dtype=F64, requires_grad=True)
        st["b"] = st["b"].clone().requires_grad_(True)
    return st


def run(state):
    S, case = state["solver"], state["case"]
    if case["api"] == "train":
        x = G.solve_differentiable(S, state["b"], state["lam"], case["iters"])
        loss = (x - state["x_true"]).square().sum()
        gb, gl = torch.autograd.grad(loss, (state["b"], state["lam"]))
        return {"x": x.detach(), "db": gb, "dlam": gl}
    S.reset(state["b"])
    if case["api"] == "batch":
        rep = S.solve(case["iters"], x_out=state["rows"])
        return {"x": state["x"], "iters": [r["iters_done"] for r in rep[:1]]}
    rep = S.solve(case["iters"], x_out=state["x"])
    return {"x": state["x"], "iters": rep["iters_done"]}


# --------------------------------------------------------------------------------------- work

def _sizes(case, frames, k):
    """(n, m, p, stored entries, operations of one A pass per vector) of one operator."""
    N, fam = case["n"], case["family"]
    ny = 1 if fam == "deconv" else case["ny"]
    n = N * ny * frames
    if fam == "deconv":
        return n, n, n - 1, n * n, 2 * n * n
    if fam == "deblur":
        return n, n, 2 * n - N - ny, 0, 2 * 81 * n
    if fam == "seismic":
        h = case["sides"]
        y = (np.arange(h) + 0.5) * (N / h)
        nnz = np.sum(N + np.abs(y[:, None] - y[None, :])) + np.sum(y[None, :] + N - y[:, None])
        return n, 2 * h * h, n, int(nnz), 2 * int(nnz)
    nnz = int(4 / math.pi * case["views"] * N * N) * frames
    return n, case["views"] * case["bins"] * frames, (2 * N * N - 2 * N) * frames + (frames - 1) * N * N, nnz, 2 * nnz


def work(case):
    """Per iteration: one read of A and one of its transpose (of the transpose again for every
    refinement step), the basis and its image read once for x and the residual (once more for every
    refinement step), the appended columns, and a dense sketch where there is one; the setup's five
    operator passes; the derivative as one more sweep of the same."""
    by = fl = 0.0
    B, F, K, R = case["batch"], case["frames"], case["iters"], case["refine"]
    groups = [(F, (B + 1) // 2), (max(2, F // 2), B // 2)] if case["family"] == "dynct" and B > 1 else [(F, B)]
    for frames, k in groups:
        n, m, p, nnz, fa = _sizes(case, frames, k)
        entry = 4 if case["family"] == "deconv" else 8
        ew, ea = (4 if case["precision"] == "fp32" else 8), 8
        cols = K * ELL + K * (K + 1) / 2
        by += nnz * entry * ((2 + R) * K + 5)
        by += k * (cols * (n * ew + m * ea) * (1 + 2 * R) + K * (n * ew + m * ea + 2 * n * 8))
        fl += k * (fa * ((2 + R) * K + 5) + cols * 2 * (n + m) * (1 + 2 * R))
        if case["sketch"] != "sparse_sign":
            by += 8.0 * case["s"] * (m + p) * K
            fl += 2.0 * case["s"] * (m + p) * K
        if case["method"] == "gks":
            by += cols * 2 * (m + p + n) * 8
            fl += cols * 8 * (m + p + n)
        if case["api"] == "train":
            by, fl = 3 * by, 3 * fl
    return {"bytes": by, "flops": fl}


# -------------------------------------------------------------------------------------- exact

class _Linear(torch.autograd.Function):
    """A linear map with its adjoint, so that the derivative of a solve can be taken through it."""

    @staticmethod
    def forward(ctx, x, fwd, adj):
        ctx.maps = fwd, adj
        return fwd(x)

    @staticmethod
    def backward(ctx, g):
        fwd, adj = ctx.maps
        return _Linear.apply(g, adj, fwd), None, None


class _Map:
    def __init__(self, fwd, adj):
        self.fwd, self.adj = fwd, adj

    def __call__(self, x):
        return _Linear.apply(x, self.fwd, self.adj)

    def t(self, x):
        return _Linear.apply(x, self.adj, self.fwd)


def _matrix(M, Mt):
    return _Map(lambda x: M @ x, lambda y: Mt @ y)


def _exact_a(P):
    if P.family == "deconv":
        M = P.dense.to(F64)
        return _matrix(M, M.t().contiguous())
    if P.family == "deblur":
        psf = P.psf.to(F64)
        img = lambda x: x.t().reshape(-1, P.ny, P.nx)  # noqa: E731
        back = lambda y: y.reshape(y.shape[0], -1).t().contiguous()  # noqa: E731
        return _Map(lambda x: back(_conv(psf, img(x))), lambda y: back(_conv(psf, img(y), True)))
    rp, col, val, m, n = P.csr
    row = torch.repeat_interleave(torch.arange(m, device=DEV), (rp[1:] - rp[:-1]).long())
    order = (col.long() * m + row).argsort()
    trp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(col.long(), minlength=n), 0, out=trp[1:])
    M = torch.sparse_csr_tensor(rp.long(), col.long(), val.to(F64), size=(m, n))
    Mt = torch.sparse_csr_tensor(trp, row[order], val.to(F64)[order], size=(n, m))
    return _matrix(M, Mt)


def _exact_l(P):
    nx, ny, nt = P.nx, P.ny, P.frames

    def diff_t(d, axis, size):
        z = torch.zeros_like(d.narrow(axis, 0, 1))
        return torch.cat([z, d], axis) - torch.cat([d, z], axis)

    if P.family == "seismic":
        def lap(x):
            u = torch.nn.functional.pad(x.t().reshape(-1, ny, nx), (1, 1, 1, 1))
            v = 4 * u[:, 1:-1, 1:-1] - u[:, :-2, 1:-1] - u[:, 2:, 1:-1] - u[:, 1:-1, :-2] - u[:, 1:-1, 2:]
            return v.reshape(x.shape[1], -1).t()
        return _Map(lap, lap)
    axes = [2] if P.family == "deconv" else [2, 1] if nt == 1 else [2, 1, 0]
    shape = (nt, ny, nx)
    parts = [[s - (a == i) for i, s in enumerate(shape)] for a in axes]

    def fwd(x):
        v = x.reshape(*shape, -1)
        return torch.cat([v.diff(dim=a).reshape(-1, x.shape[1]) for a in axes])

    def adj(d):
        out, at = 0, 0
        for a, q in zip(axes, parts):
            c = q[0] * q[1] * q[2]
            out = out + diff_t(d[at:at + c].reshape(*q, -1), a, shape[a])
            at += c
        return out.reshape(-1, d.shape[1])

    return _Map(fwd, adj)


def _mix(z):
    with np.errstate(over="ignore"):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))


def _sparse_sign(seed, stream, h, s):
    """Column j of the sketch: ZETA distinct rows and signs from the counter-based hash of (seed,
    stream, j, draw), a repeated row skipped."""
    key = _mix(np.uint64(2 * int(seed) + stream))
    rows, signs, have = np.full((h, ZETA), -1, np.int64), np.zeros((h, ZETA)), np.zeros(h, np.int64)
    for c in range(256):
        j = np.flatnonzero(have < ZETA)
        if not j.size:
            break
        hv = _mix(key ^ ((j.astype(np.uint64) << np.uint64(8)) | np.uint64(c)))
        r = (((hv >> np.uint64(32)) * np.uint64(s)) >> np.uint64(32)).astype(np.int64)
        new = ~(rows[j] == r[:, None]).any(1)
        rows[j[new], have[j[new]]] = r[new]
        signs[j[new], have[j[new]]] = np.where(hv[new] & np.uint64(1), -1.0, 1.0) / math.sqrt(ZETA)
        have[j[new]] += 1
    row = torch.from_numpy(rows.reshape(-1)).to(DEV)
    col = torch.arange(h, device=DEV).repeat_interleave(ZETA)
    val = torch.from_numpy(signs.reshape(-1)).to(DEV)
    order = (row * h + col).argsort()
    rp = torch.zeros(s + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(row, minlength=s), 0, out=rp[1:])
    cp = torch.arange(0, ZETA * h + 1, ZETA, device=DEV)
    by = (col * s + row).argsort()
    return _matrix(torch.sparse_csr_tensor(rp, col[order], val[order], size=(s, h)),
                   torch.sparse_csr_tensor(cp, row[by], val[by], size=(h, s)))


def _exact_sketch(case, seed, P):
    m, p, s = P.m, P.p(), case["s"]
    if case["method"] == "gks":
        same = _Map(lambda x: x, lambda x: x)
        return same, same
    if case["sketch"] == "sparse_sign":
        sk = int(seed) & 0x7FFFFFFF
        return _sparse_sign(sk, 0, m, s), _sparse_sign(sk, 1, p, s)
    got = _sketch_inputs(case, seed, m, p)
    if case["sketch"] == "gaussian":
        return tuple(_matrix(M, M.t()) for M in got)
    maps = []
    for h, signs, rows in ((m, got[0], got[1]), (p, got[2], got[3])):
        k, i = rows.long()[:, None], torch.arange(h, device=DEV)[None, :]
        M = torch.cos(((k * (2 * i + 1)) % (4 * h)).to(F64) * (math.pi / (2 * h))) * signs.to(F64)[None, :]
        M *= math.sqrt(h / s) * torch.where(k == 0, math.sqrt(1.0 / h), math.sqrt(2.0 / h)).to(F64)
        maps.append(_matrix(M, M.t()))
    return tuple(maps)


def _project(cols, v, times=2):
    """Classical Gram-Schmidt of v [h, k] against orthonormal columns, `times` passes: (v, coefficients)."""
    if not cols:
        return v, v.new_zeros(0, v.shape[1])
    Q, c = torch.stack(cols), 0
    for _ in range(times):
        d = (Q * v).sum(1)
        v = v - (Q * d[:, None, :]).sum(0)
        c = c + d
    return v, c


def _exact_solve(case, seed, P, b, lam):
    """Algorithm 2 (or 1) for the k right-hand sides b [m, k], lam [k] at once, in float64."""
    A, L, (SA, SL) = _exact_a(P), _exact_l(P), _exact_sketch(case, seed, P)
    gks, k = case["method"] == "gks", b.shape[1]
    zero = b.new_zeros(L(b.new_zeros(P.n, k)).shape) if gks else b.new_zeros(case["s"], k)
    rhs = torch.cat([SA(b), zero])
    W, Q, R, c = [], [], [], []

    def append(w):
        W.append(w)
        v, p = _project(Q, torch.cat([SA(A(w)), lam.sqrt() * SL(L(w))]))
        rho = v.norm(dim=0)
        Q.append(v / rho)
        R.append(torch.cat([p, rho[None]]))
        c.append((Q[-1] * rhs).sum(0))

    def solve_t(g, transposed):
        d = len(R)
        y = [None] * d
        for i in (range(d) if transposed else reversed(range(d))):
            r = g[i]
            for j in (range(i) if transposed else range(i + 1, d)):
                r = r - (R[i][j] if transposed else R[j][i]) * y[j]
            y[i] = r / R[i][i]
        return y

    def combine(y):
        x = W[0] * y[0]
        for w, t in zip(W[1:], y[1:]):
            x = x + w * t
        return x

    def gradient(x):
        return A.t(A(x) - b) + lam * L.t(L(x))

    v = A.t(b)
    V = [v / v.norm(dim=0)]
    while len(V) < ELL:
        v, _ = _project(V, A.t(A(V[-1])))
        V.append(v / v.norm(dim=0))
    for v in V:
        append(v)
    for it in range(case["iters"] + 1):
        y = solve_t(c, False)
        for _ in range(case["refine"]):
            r = gradient(combine(y))
            d = solve_t(solve_t([(w * r).sum(0) for w in W], True), False)
            y = [a - e for a, e in zip(y, d)]
        x = combine(y)
        if it == case["iters"]:
            return x
        r = gradient(x)
        if gks:
            r, _ = _project(W, r)
            r = r / r.norm(dim=0)
        append(r)


def exact(case, seed):
    probs = _problems(case, seed)
    if case["api"] == "train":
        P = probs[0]
        b = P.b[0].clone().requires_grad_(True)
        lam = torch.tensor([P.lam[0]], dtype=F64, device=DEV, requires_grad=True)
        x = _exact_solve(case, seed, P, b[:, None], lam)[:, 0]
        gb, gl = torch.autograd.grad((x - P.x_true).square().sum(), (b, lam))
        return {"x": x.detach(), "db": gb, "dlam": gl[0]}
    with torch.no_grad():
        xs = []
        for P in probs:
            lam = torch.tensor(P.lam, dtype=F64, device=DEV)
            part = max(1, (8 << 30) // (8 * P.n * (case["iters"] + ELL)))
            xs.append(torch.cat([_exact_solve(case, seed, P, torch.stack(P.b[i:i + part], 1), lam[i:i + part]).t()
                                 for i in range(0, len(P.b), part)]))
    if case["api"] == "batch":
        return {"x": xs, "iters": [None]}
    return {"x": xs[0][0], "iters": None}
