"""Timed cases of the AIR library: single operators, whole solves, a batch and a served queue.

A case is one call (or, for the server, one queue of requests) through the
public binding ``paper_1310_1434_gb300.air``.  Geometries are those of
``paper_1310_1434_gb300.inputs`` (128, 256, 512 and 1024 pixels over about
410 mm), of the tests' ragged shapes, and the paper's 350 x 350 x 1 mm, 528
bins, 800 or 200 views.  Sinograms are line integrals of random ellipse
phantoms with Poisson counting noise, images are such phantoms rasterised.

``exact`` evaluates the same operators in 64 bits with plain torch: explicit
ray-pixel lengths, an FFT filter, framelets by rolls, and CG on them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1310_1434_gb300 import air, inputs

DEV = "cuda"
DSO = 850.0
FBS_STEP = 0.6          # below 1 / ||A^T C A||, which is near 1 at these geometries


# ------------------------------------------------------------------ cases --
def _op(name, op, n, px, views, bins, prec=0, **kw):
    return dict(name=name, op=op, n=n, px=px, views=views, bins=bins, prec=prec, **kw)


def listed():
    return [
        # the projector on the smallest configuration: a call of a user's own
        # iteration on a scout image, where latency and launches count
        _op("project_128_v90", "project", 128, 1.0, 90, 192),
        # the projector at the main configuration: the data term of one slice
        _op("project_512_v800", "project", 512, 0.8, 800, 738),
        # the exact adjoint on the paper's own image and 25 % data: a ragged
        # image side (350 = 10 tiles and 30 pixels)
        _op("backproject_350_v200", "backproject", 350, 1.0, 200, 528),
        # the filtered adjoint A^T C of the largest served slice, FP32 filter
        _op("fbackproject_1024_v800", "fbackproject", 1024, 0.4, 800, 1476),
        # the ramp filter on tensor cores at the main configuration
        _op("filter_bf16x3_512_v800", "filter", 512, 0.8, 800, 738, prec=1),
        # one d/b update of the split-Bregman loop, for a user's own solver
        _op("shrink_512", "shrink", 512, 0.8, 16, 64, tau=3e-4),
        # the analytic reconstruction the paper compares with, its geometry
        _op("fbp_350_v800", "fbp", 350, 1.0, 800, 528),
        # a whole solve of the smallest configuration, FP32
        _op("solve_128_v90", "solve", 128, 1.0, 90, 192, lam=0.01, outer=20, cg=5),
        # a whole solve of one main-configuration slice, split-BF16 filter
        _op("solve_512_v800_bf16x3", "solve", 512, 0.8, 800, 738, prec=1, lam=3e-4, outer=30, cg=8),
        # forward-backward splitting of a quick-look slice, FP32
        _op("fbs_256_v200", "fbs", 256, 1.6, 200, 384, lam=3e-4, iters=60),
        # the batched form the throughput figure is quoted on: eight slices,
        # full and 25 % view counts in turn
        dict(name="batch_8x512", op="batch", prec=1, lam=3e-4, outer=30, cg=8,
             slices=" ".join(["512:0.8:800:738", "512:0.8:200:738"] * 4)),
        # a served queue of uneven requests, from and to host memory
        dict(name="serve_6_uneven", op="serve", prec=0, lam=3e-4, outer=30, cg=8,
             slices="256:1.6:200:384 512:0.8:200:738 512:0.8:400:738 256:1.6:800:384 "
                    "1024:0.4:200:1476 256:1.6:400:384"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_slice(rng, lo=64, hi=1024, vmax=800):
    n = _log_int(rng, lo, hi)
    px = round(409.6 / n, 4) if rng.random() < 0.7 else round(rng.uniform(0.5, 1.0) * 409.6 / n, 4)
    return n, px, _log_int(rng, 45, vmax), int(n * rng.uniform(1.25, 1.6)) + 1


def _spec(s):
    return "%d:%r:%d:%d" % s


def draw(rng):
    op = rng.choice(["project", "backproject", "fbackproject", "filter", "shrink", "fbp", "solve", "l2", "fbs",
                     "batch", "serve"])
    prec = rng.randint(0, 1)
    if op in ("batch", "serve"):
        sl = [_draw_slice(rng, 64, 512, 400) for _ in range(rng.randint(2, 6))]
        return dict(op=op, prec=prec, lam=3e-4, outer=rng.randint(3, 12), cg=rng.randint(3, 8),
                    slices=" ".join(_spec(s) for s in sl))
    n, px, views, bins = _draw_slice(rng)
    case = dict(op=op, n=n, px=px, views=views, bins=bins, prec=prec)
    if op == "shrink":
        case.update(tau=10.0 ** rng.uniform(-4, -2))
    if op == "solve":
        case.update(lam=10.0 ** rng.uniform(-4, -2), outer=rng.randint(2, 12), cg=rng.randint(3, 8))
    if op == "l2":
        case.update(lam=10.0 ** rng.uniform(-2, 0), iters=rng.randint(5, 60))
    if op == "fbs":
        case.update(lam=10.0 ** rng.uniform(-4, -3), iters=rng.randint(5, 60))
    return case


def _slices(case):
    """The (n, px, views, bins) of a case's slices."""
    if "slices" in case:
        out = []
        for s in case["slices"].split():
            n, px, views, bins = s.split(":")
            out.append((int(n), float(px), int(views), int(bins)))
        return out
    return [(case["n"], case["px"], case["views"], case["bins"])]


def _geom(sl, prec):
    n, px, views, bins = sl
    return inputs.Geometry(n, px, views, bins, dso_mm=DSO, precision=prec)


# ----------------------------------------------------------------- inputs --
def _rays(g):
    """Source points (V, 1) and unit directions (V, bins) of every ray, 64 bits."""
    beta = g.beta0 + g.arc * torch.arange(g.n_views, dtype=torch.float64, device=DEV)[:, None] / g.n_views
    gamma = (torch.arange(g.n_bins, dtype=torch.float64, device=DEV) - 0.5 * (g.n_bins - 1)) * g.fan_pitch
    th = beta + math.pi + gamma[None, :]
    return g.dso_mm * torch.cos(beta), g.dso_mm * torch.sin(beta), torch.cos(th), torch.sin(th)


def _sinogram(g, seed, photons=2e4):
    """A measured sinogram (V, bins) in FP32: exact ellipse line integrals, counting noise."""
    sx, sy, ux, uy = _rays(g)
    p = torch.zeros(g.n_views, g.n_bins, dtype=torch.float64, device=DEV)
    for e in inputs.random_phantom(g, seed, 8, 4):
        rx, ry = sx - e.cx, sy - e.cy
        t = rx * ux + ry * uy
        rx, ry = rx - t * ux, ry - t * uy
        c, s = math.cos(e.phi), math.sin(e.phi)
        qx, qy, wx, wy = rx * c + ry * s, ry * c - rx * s, ux * c + uy * s, uy * c - ux * s
        A = wx * wx / e.a ** 2 + wy * wy / e.b ** 2
        B = qx * wx / e.a ** 2 + qy * wy / e.b ** 2
        C = qx * qx / e.a ** 2 + qy * qy / e.b ** 2 - 1.0
        p += 2.0 * e.rho * torch.sqrt(torch.clamp(B * B - A * C, min=0.0)) / A
    gen = torch.Generator(device=DEV).manual_seed(seed + 0x5EED)
    counts = torch.poisson(photons * torch.exp(-p), generator=gen)
    return (-torch.log(torch.clamp(counts, min=1.0) / photons)).float()


def _image(g, seed):
    """A phantom image (n, n) in FP32 with a little noise, as an iterate has it."""
    n, dx = g.n, g.pixel_mm
    c = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5 - 0.5 * n) * dx
    x, y = c[None, :], c[:, None]
    X = torch.zeros(n, n, dtype=torch.float64, device=DEV)
    for e in inputs.random_phantom(g, seed, 8, 4):
        co, s = math.cos(e.phi), math.sin(e.phi)
        u, v = (x - e.cx) * co + (y - e.cy) * s, (y - e.cy) * co - (x - e.cx) * s
        X += e.rho * ((u / e.a) ** 2 + (v / e.b) ** 2 <= 1.0)
    gen = torch.Generator(device=DEV).manual_seed(seed + 77)
    X += 4e-4 * torch.randn(n, n, dtype=torch.float64, device=DEV, generator=gen)
    return X.float()


def _bregman(n, tau, seed):
    """A Bregman variable (9, n, n) as the loop leaves it: within the threshold, zero on band 0."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 99)
    b = (torch.rand(9, n, n, device=DEV, generator=gen) * 2.0 - 1.0) * tau
    b[0] = 0.0
    return b


def _inputs(case, seed):
    """The data of a case, on the device: a list with one tensor for each slice (shrink: X and b)."""
    op = case["op"]
    gs = [_geom(s, case["prec"]) for s in _slices(case)]
    seeds = [1000 * seed + 17 * i for i in range(len(gs))]
    if op == "project":
        return gs, [_image(gs[0], seeds[0])]
    if op == "shrink":
        return gs, [_image(gs[0], seeds[0]), _bregman(gs[0].n, case["tau"], seeds[0])]
    return gs, [_sinogram(g, s) for g, s in zip(gs, seeds)]


def prepare(case, seed):
    op = case["op"]
    gs, data = _inputs(case, seed)
    st = {"case": case, "op": op, "data": data}
    if op == "serve":
        st["geoms"] = gs
        st["host"] = [y.cpu().numpy() for y in data]
        st["server"] = air.Server(32 << 30, 16)
        return st
    st["plans"] = [air.Plan(g) for g in gs]
    g = gs[0]
    if op in ("project", "filter"):
        st["out"] = torch.empty(g.n_views, g.n_bins, device=DEV)
    else:
        st["out"] = [torch.empty(q.n, q.n, device=DEV) for q in gs]
    if op == "shrink":
        st["resid"] = torch.zeros(1, dtype=torch.float64, device=DEV)
    if op == "solve":
        st["resid"] = torch.zeros(case["outer"], dtype=torch.float64, device=DEV)
    return st


def run(st):
    case, op, data = st["case"], st["op"], st["data"]
    if op == "serve":
        srv = st["server"]
        ids = [srv.submit(g, y, case["lam"], 1.0, case["outer"], case["cg"]) for g, y in zip(st["geoms"], st["host"])]
        return [srv.wait(i) for i in ids]
    out = st["out"]
    if op == "batch":
        k = len(data)
        air.air_solve_batch(st["plans"], data, [case["lam"]] * k, [1.0] * k, [case["outer"]] * k, [case["cg"]] * k, out)
        return out
    plan, x = st["plans"][0], data[0]
    if op == "project":
        air.air_project(plan, x, out)
        return out
    if op == "filter":
        air.air_filter(plan, x, out)
        return out
    X = out[0]
    if op == "backproject":
        air.air_backproject(plan, x, X)
    elif op == "fbackproject":
        air.air_filtered_backproject(plan, x, X)
    elif op == "fbp":
        air.air_fbp(plan, x, X)
    elif op == "shrink":
        air.air_shrink(plan, x, data[1], X, case["tau"], st["resid"])
        return [data[1], X, st["resid"]]
    elif op == "solve":
        air.air_solve(plan, x, case["lam"], 1.0, case["outer"], case["cg"], X, st["resid"])
        return [X, st["resid"]]
    elif op == "l2":
        air.air_solve_l2(plan, x, case["lam"], case["iters"], X)
    elif op == "fbs":
        air.air_solve_fbs(plan, x, case["lam"], FBS_STEP, case["iters"], X)
    return X


def work(case):
    """Inputs and results once; two operations for each ray-pixel length, an FFT's for each filtered row."""
    op, nbytes, flops = case["op"], 0.0, 0.0
    for n, _, views, bins in _slices(case):
        image, sino = 4.0 * n * n, 4.0 * views * bins
        ray = 2.0 * 0.89 * n * views * bins           # 0.89 n lengths on a ray, the mean over the fan
        fft = 10.0 * views * bins * math.log2(2.0 * bins)
        vec = 60.0 * n * n                            # one shrink: 9 bands both ways
        if op == "shrink":
            nbytes, flops = nbytes + 2 * image + 18 * image, flops + vec
            continue
        nbytes += sino if op == "filter" else image
        nbytes += sino
        pairs = {"solve": case.get("outer", 0) * case.get("cg", 0), "batch": case.get("outer", 0) * case.get("cg", 0),
                 "serve": case.get("outer", 0) * case.get("cg", 0), "l2": case.get("iters", 0),
                 "fbs": case.get("iters", 0)}.get(op)
        if pairs is not None:
            flops += pairs * (2 * ray + fft + 10.0 * n * n) + ray + fft
            flops += vec * (case["outer"] if "outer" in case else pairs if op == "fbs" else 0)
        elif op == "project" or op == "backproject":
            flops += ray
        elif op == "filter":
            flops += fft
        elif op == "fbackproject":
            flops += ray + fft
        elif op == "fbp":
            flops += fft + 12.0 * n * n * views
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------ 64-bit values --
def _chunks(g):
    step = max(1, int(2 ** 26 / (g.n_bins * g.n)))
    return [(v, min(g.n_views, v + step)) for v in range(0, g.n_views, step)]


def _lengths(g, v0, v1):
    """Pixels (rays, 2 n) and lengths in mm of the rays of views [v0, v1), zero length where there is none."""
    n, dx = g.n, g.pixel_mm
    sx, sy, ux, uy = (t[v0:v1] for t in _rays(g))
    t = sx * ux + sy * uy
    px, py = ((sx - t * ux) / dx + 0.5 * n).reshape(-1), ((sy - t * uy) / dx + 0.5 * n).reshape(-1)
    ux, uy = ux.reshape(-1), uy.reshape(-1)
    cols = ux.abs() >= uy.abs()
    a, b = torch.where(cols, px, py), torch.where(cols, py, px)
    ua, ub = torch.where(cols, ux, uy), torch.where(cols, uy, ux)
    m = ub / ua
    k = torch.arange(n, dtype=torch.float64, device=DEV)[None, :]
    # a ray on a grid line belongs to the upper side
    lo = (b - a * m)[:, None] + m[:, None] * k + torch.clamp(m, max=0.0)[:, None] + 1e-9
    am = m.abs()[:, None]
    r = torch.floor(lo)
    sec = (dx / ua.abs())[:, None]
    first = torch.where(am > 1e-12, torch.clamp((r + 1.0 - lo) / torch.clamp(am, min=1e-12), max=1.0), torch.ones_like(lo))
    ki, ri = k.long().expand_as(lo), r.long()
    pix, val = [], []
    for row, w in ((ri, first * sec), (ri + 1, (1.0 - first) * sec)):
        ok = (row >= 0) & (row < n)
        row = row.clamp(0, n - 1)
        pix.append(torch.where(cols[:, None], row * n + ki, ki * n + row))
        val.append(torch.where(ok, w, torch.zeros_like(w)))
    return torch.cat(pix, 1), torch.cat(val, 1)


def _A(g, X):
    X = X.double().reshape(-1)
    out = [(val * X[pix]).sum(1) for pix, val in (_lengths(g, *c) for c in _chunks(g))]
    return torch.cat(out).reshape(g.n_views, g.n_bins)


def _AT(g, Y):
    X = torch.zeros(g.n * g.n, dtype=torch.float64, device=DEV)
    for v0, v1 in _chunks(g):
        pix, val = _lengths(g, v0, v1)
        X.index_add_(0, pix.reshape(-1), (val * Y[v0:v1].double().reshape(-1, 1)).reshape(-1))
    return X.reshape(g.n, g.n)


def _csr(rows, cols, vals, shape):
    """A sparse matrix from entries already in row order."""
    ptr = torch.zeros(shape[0] + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=shape[0]), 0)
    return torch.sparse_csr_tensor(ptr.int(), cols.int(), vals, shape)


def _matrices(g):
    """A and A^T as sparse matrices, for solves that apply them often."""
    rows, cols, vals = [], [], []
    for v0, v1 in _chunks(g):
        pix, val = _lengths(g, v0, v1)
        i, j = torch.nonzero(val, as_tuple=True)
        rows.append((i + v0 * g.n_bins).int())
        cols.append(pix[i, j].int())
        vals.append(val[i, j])
    rows, cols, vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
    A = _csr(rows, cols, vals, (g.n_views * g.n_bins, g.n * g.n))
    cols, order = torch.sort(cols, stable=True)
    return A, _csr(cols, rows[order], vals[order], (g.n * g.n, g.n_views * g.n_bins))


def _convolve(Y, taps):
    """Rows of Y convolved with the symmetric taps (lags 0 .. bins - 1), linear."""
    nb = Y.shape[1]
    L = 1 << (2 * nb - 1).bit_length()
    h = torch.zeros(L, dtype=torch.float64, device=DEV)
    h[:nb] = taps
    h[L - nb + 1:] = taps[1:].flip(0)
    return torch.fft.irfft(torch.fft.rfft(Y.double(), n=L) * torch.fft.rfft(h), n=L)[:, :nb]


def _C(g, Y):
    k = torch.arange(g.n_bins, dtype=torch.float64, device=DEV)
    h = torch.where(k % 2 == 1, -1.0 / (math.pi * torch.clamp(k, min=1.0)) ** 2, torch.zeros_like(k))
    h[0] = 0.25
    return _convolve(Y, h * (math.pi / (g.n_views * g.pixel_mm ** 2)))


_FRAME = ((0.25, 0.5, 0.25), (math.sqrt(2.0) / 4.0, 0.0, -math.sqrt(2.0) / 4.0), (-0.25, 0.5, -0.25))


def _W(X):
    out = []
    for a in _FRAME:
        R = sum(a[p + 1] * torch.roll(X, -p, 0) for p in (-1, 0, 1))
        out += [sum(b[q + 1] * torch.roll(R, -q, 1) for q in (-1, 0, 1)) for b in _FRAME]
    return torch.stack(out)


def _WT(D):
    X = 0.0
    for i, a in enumerate(_FRAME):
        for j, b in enumerate(_FRAME):
            R = sum(b[q + 1] * torch.roll(D[3 * i + j], q, 1) for q in (-1, 0, 1))
            X = X + sum(a[p + 1] * torch.roll(R, p, 0) for p in (-1, 0, 1))
    return X


def _soft(D, tau):
    S = torch.sign(D) * torch.clamp(D.abs() - tau, min=0.0)
    S[0] = D[0]
    return S


def _shrink(X, b, tau):
    w = _W(X)
    t = w + b
    d = _soft(t, tau)
    return t - d, _WT(2.0 * d - t), torch.linalg.vector_norm(w - d).reshape(1)


def _cg(M, rhs, X, steps):
    r = rhs - M(X)
    p, rho = r, (r * r).sum()
    for _ in range(steps):
        if float(rho) == 0.0:
            break
        q = M(p)
        pq = (p * q).sum()
        if not float(pq) > 0.0:
            break
        X, r = X + rho / pq * p, r - rho / pq * q
        new = (r * r).sum()
        p, rho = r + new / rho * p, new
    return X


def _solve(g, mats, Y, case):
    """The image of a solve and, for the split-Bregman form, its residual history."""
    A, AT = mats

    def adj(s):
        return (AT @ _C(g, s).reshape(-1)).reshape(g.n, g.n)

    def normal(X):
        return adj((A @ X.reshape(-1)).reshape(g.n_views, g.n_bins))

    rhs0 = adj(Y.double())
    X = torch.zeros(g.n, g.n, dtype=torch.float64, device=DEV)
    if case["op"] == "l2":
        return _cg(lambda p: normal(p) + case["lam"] * p, rhs0, X, case["iters"]), None
    if case["op"] == "fbs":
        for _ in range(case["iters"]):
            X = _WT(_soft(_W(X + FBS_STEP * (rhs0 - normal(X))), FBS_STEP * case["lam"]))
        return X, None
    b, gg, hist = torch.zeros(9, g.n, g.n, dtype=torch.float64, device=DEV), torch.zeros_like(X), []
    for _ in range(case["outer"]):
        X = _cg(lambda p: normal(p) + p, rhs0 + gg, X, case["cg"])
        b, gg, r = _shrink(X, b, case["lam"])
        hist.append(r)
    return X, torch.cat(hist)


def _fbp(g, Y):
    n, D, al = g.n, g.dso_mm, g.fan_pitch
    jm = 0.5 * (g.n_bins - 1)
    k = torch.arange(g.n_bins, dtype=torch.float64, device=DEV)
    h = torch.where(k % 2 == 1, -1.0 / (2.0 * math.pi ** 2 * torch.sin(torch.clamp(k, min=1.0) * al) ** 2), torch.zeros_like(k))
    h[0] = 1.0 / (8.0 * al * al)
    Q = _convolve(Y.double() * torch.cos((k - jm) * al), al * D * h)
    Q = torch.nn.functional.pad(Q, (1, 2))                    # zero beyond the detector
    c = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5 - 0.5 * n) * g.pixel_mm
    x, y = c[None, :], c[:, None]
    X = torch.zeros(n, n, dtype=torch.float64, device=DEV)
    for v in range(g.n_views):
        beta = g.beta0 + g.arc * v / g.n_views
        cx, cy = -math.cos(beta), -math.sin(beta)
        cr, dt = cx * y - cy * x, D + cx * x + cy * y
        t = torch.atan2(cr, dt) / al + jm
        j = torch.floor(t)
        i = (j.long() + 1).clamp(0, g.n_bins + 1)
        inside = (j >= -1) & (j < g.n_bins)
        w = t - j
        X += torch.where(inside, (1.0 - w) * Q[v][i] + w * Q[v][i + 1], torch.zeros_like(w)) / (cr * cr + dt * dt)
    return X * (g.arc / g.n_views)


def exact(case, seed):
    op = case["op"]
    gs, data = _inputs(case, seed)
    g, x = gs[0], data[0]
    if op == "project":
        return _A(g, x)
    if op == "filter":
        return _C(g, x)
    if op == "backproject":
        return _AT(g, x)
    if op == "fbackproject":
        return _AT(g, _C(g, x))
    if op == "fbp":
        return _fbp(g, x)
    if op == "shrink":
        b, u, r = _shrink(x.double(), data[1].double(), case["tau"])
        return [b, u, r]
    mats, out = {}, []
    for q, y in zip(gs, data):
        key = (q.n, q.pixel_mm, q.n_views, q.n_bins)
        if key not in mats:
            if len(mats) > 2:
                mats.clear()
            mats[key] = _matrices(q)
        out.append(_solve(q, mats[key], y, case))
    if op == "serve":
        return [X.reshape(-1).cpu().numpy() for X, _ in out]
    if op == "batch":
        return [X for X, _ in out]
    return out[0][0] if op != "solve" else list(out[0])
