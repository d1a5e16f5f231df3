"""The calls this framework is measured on: one pass of each through the public
Python entry points, with the inputs a program has in hand before the call.

``listed()`` are the fixed cases, ``draw(rng)`` gives one more of the same
ranges, ``prepare`` makes a case's inputs from a seed, ``run`` is one pass,
``work`` the bytes and operations a pass cannot do without, ``exact`` the
outputs in plain 64-bit arithmetic where they can be had in seconds.

Kinds and what they stand for in use:

* split      one split step of a caller's own time loop on a small grid: the
             smallest call, all latency
* solve      one stationary solve to tolerance on a handle that is kept (other
             loads on the same domain would reuse it): small, ordinary and
             large grids, FP64 and FP32 + refinement, the transfer through the
             grid and the direct one, the plain and the accelerated iteration
* new        a problem met for the first time: setup, solve and release
* slices     implicit-Euler time steps, each slice solved to tolerance
* steps      the paper's own time stepping, one split step per time step
* batch      many independent problems of uneven size and shape in one launch
* forward    the warm-start network's prediction for a batch of problems
* gradient   loss and gradients of a training batch of that network
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2411_11041_gb300 as adr
from paper_2411_11041_gb300 import workloads as W

DEV = "cuda:0"
HW = 64  # network cells per side


def listed():
    return [
        # latency of a single call on the 64 x 64 manufactured problem
        dict(name="split64", kind="split", field="slant", nx=64, ny=64),
        # the 64 x 64 manufactured configuration, solved to 1e-10
        dict(name="solve64", kind="solve", field="slant", nx=64, ny=64, tol=1e-10, prec=0, transfer=0,
             anderson=0),
        # the paper's experiment: 50 Crank-Nicolson steps of 1e-3 on a rotating field
        dict(name="paper61", kind="steps", field="rotating", nx=61, ny=61, dt=1e-3, nsteps=50),
        # an ordinary single problem, curved flow
        dict(name="solve513", kind="solve", field="sheared", nx=513, ny=513, tol=1e-8, prec=0, transfer=0,
             anderson=0),
        # the headline problem: 2048 x 2048, advection dominated
        dict(name="solve2048", kind="solve", field="sheared", nx=2048, ny=2048, tol=1e-8, prec=0, transfer=0,
             anderson=0),
        # FP32 line solves with FP64 refinement, one node off a power of two
        dict(name="refine1025", kind="solve", field="sheared", nx=1025, ny=1025, tol=1e-8, prec=1, transfer=0,
             anderson=0),
        # values carried from curve to curve, on a rectangle of odd sizes
        dict(name="direct1501", kind="solve", field="sheared", nx=1501, ny=1333, tol=1e-8, prec=0, transfer=1,
             anderson=0),
        # the first implicit-Euler steps of the 1024 x 1024 blob, accelerated
        dict(name="slices1024", kind="slices", field="sheared", nx=1024, ny=1024, tol=1e-8, dt=1e-3, nsteps=4,
             anderson=3),
        # setup + solve of one problem met for the first time
        dict(name="new1024", kind="new", field="sheared", nx=1024, ny=1024, tol=1e-8),
        # a batch of uneven problems: sizes 128 to 1024, squares, discs and L shapes
        dict(name="batch48", kind="batch", count=48, nmin=128, nmax=1024, tol=1e-8, prec=0, anderson=0, base=0),
        # prediction for 128 problems
        dict(name="forward128", kind="forward", batch=128),
        # one training batch
        dict(name="gradient64", kind="gradient", batch=64),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["split", "solve", "solve", "solve", "steps", "slices", "new", "batch", "forward",
                       "gradient"])
    if kind == "split":
        return dict(kind=kind, field="slant", nx=_logint(rng, 33, 700), ny=_logint(rng, 33, 700))
    if kind == "solve":
        n = _logint(rng, 48, 2048)
        transfer = rng.choice([0, 0, 0, 1])
        prec = 0 if transfer else rng.choice([0, 0, 1])
        anderson = 0 if prec else rng.choice([0, 0, 0, 2])
        return dict(kind=kind, field=rng.choice(["slant", "sheared", "sheared"]), nx=n,
                    ny=max(40, min(2048, int(n * rng.uniform(0.7, 1.3)))), tol=rng.choice([1e-8, 1e-10]),
                    prec=prec, transfer=transfer, anderson=anderson)
    if kind == "steps":
        n = _logint(rng, 40, 600)
        return dict(kind=kind, field=rng.choice(["rotating", "sheared"]), nx=n, ny=n,
                    dt=rng.choice([1e-3, 2e-3]), nsteps=rng.randint(10, 60))
    if kind == "slices":
        n = _logint(rng, 64, 1024)
        return dict(kind=kind, field="sheared", nx=n, ny=n, tol=1e-8, dt=1e-3, nsteps=rng.randint(1, 4),
                    anderson=rng.choice([0, 3]))
    if kind == "new":
        n = _logint(rng, 64, 1024)
        return dict(kind=kind, field=rng.choice(["slant", "sheared"]), nx=n, ny=n, tol=1e-8)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 32), nmin=rng.randint(64, 128),
                    nmax=rng.randint(200, 800), tol=1e-8, prec=rng.choice([0, 1]), anderson=0,
                    base=rng.randint(1, 1000))
    return dict(kind=kind, batch=_logint(rng, 1, 128 if kind == "forward" else 64))


# ------------------------------------------------------------------ inputs

def _coords(nx, ny, y1):
    x = torch.arange(nx, dtype=torch.float64, device=DEV) / (nx - 1)
    y = y1 * torch.arange(ny, dtype=torch.float64, device=DEV) / (ny - 1)
    return x[None, :].expand(ny, nx), y[:, None].expand(ny, nx)


def _sources(nx, ny, y1, centres):
    """Sum of unit Gaussians of width 0.02 at the centres (the workloads' source)."""
    X, Y = _coords(nx, ny, y1)
    f = torch.zeros((ny, nx), dtype=torch.float64, device=DEV)
    for cx, cy in centres:
        f += torch.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / (2.0 * W.GAUSS_WIDTH ** 2))
    return f


def _centres(rng, y1=1.0):
    c = rng.uniform(0.1, 0.9, size=(W.N_GAUSS, 2))
    return c * np.array([1.0, y1])


def _problem(case, seed):
    """Nodal data of one problem (device tensors) and its state u0, if any."""
    nx, ny, field = case["nx"], case["ny"], case["field"]
    rng = np.random.Generator(np.random.PCG64([W.SEED_BASE, seed]))
    y1 = round(ny / nx, 6) if nx != ny else 1.0
    X, Y = _coords(nx, ny, y1)
    one = torch.ones((ny, nx), dtype=torch.float64, device=DEV)
    u0 = None
    f = _sources(nx, ny, y1, _centres(rng, y1))
    if field == "slant":  # the manufactured configuration's coefficients
        mu, sigma = 0.1, 1.0
        b1, b2 = one, 0.5 * one
        f = f + rng.uniform(0.5, 2.0) * torch.sin(math.pi * X) * torch.sin(math.pi * Y / y1)
    elif field == "sheared":
        mu, sigma = 1e-3, 1.0
        b1, b2 = one, 0.5 + 0.3 * torch.sin(2.0 * math.pi * X)
        if case["kind"] in ("slices", "steps"):
            mu, sigma = 1e-2, 0.5
            f = torch.zeros_like(one)
            cx, cy = rng.uniform(0.2, 0.4), rng.uniform(0.4, 0.6)
            u0 = torch.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / (2.0 * 0.05 ** 2))
    else:  # rotating: the paper's experiment, with the load's level drawn
        mu, sigma = 1.0, 1.0
        b1, b2 = -5.0 * (Y + 1.0), 5.0 * (X + 1.0)
        f = rng.uniform(4.0, 6.0) * one + f
    mask = torch.ones((ny, nx), dtype=torch.uint8, device=DEV)
    p = W.Problem(nx, ny, mu, sigma, b1.contiguous(), b2.contiguous(), f.contiguous(), mask, y1=y1, u0=u0)
    return p


def _options(case):
    o = dict(tol=case.get("tol", 1e-8), max_iter=100000, prec=case.get("prec", 0),
             transfer=case.get("transfer", 0), anderson=case.get("anderson", 0))
    return o


def _batch_problems(case, seed):
    """Sizes, domains and coefficients belong to the case; the sources to the seed."""
    fixed = np.random.Generator(np.random.PCG64([W.SEED_BASE + 3, case["base"]]))
    rng = np.random.Generator(np.random.PCG64([W.SEED_BASE, seed]))
    out = []
    for _ in range(case["count"]):
        n = int(fixed.integers(case["nmin"], case["nmax"] + 1))
        kind = W.MASKS[int(fixed.integers(0, len(W.MASKS)))]
        mu, sigma = float(10.0 ** fixed.uniform(-4.0, -1.0)), float(fixed.uniform(0.1, 2.0))
        phi = fixed.uniform(0.0, 2.0 * math.pi)
        one = torch.ones((n, n), dtype=torch.float64, device=DEV)
        mask = torch.as_tensor(W.make_mask(kind, n, n), device=DEV)
        out.append(W.Problem(n, n, mu, sigma, math.cos(phi) * one, math.sin(phi) * one,
                             _sources(n, n, 1.0, _centres(rng)), mask))
    return out


def _net_inputs(case, seed):
    """Features as the network meets them: per 4 x 4-node cell the sources, a
    plume downstream of them (the scaled first state), and the coefficients."""
    B, n = case["batch"], 4 * HW
    rng = np.random.Generator(np.random.PCG64([W.SEED_BASE + 4, seed]))
    x = torch.zeros((B, HW, HW, 40), dtype=torch.float64, device=DEV)
    t = torch.zeros((B, HW, HW), dtype=torch.float32, device=DEV)
    X, Y = _coords(n, n, 1.0)
    for b in range(B):
        phi = rng.uniform(0.0, 2.0 * math.pi)
        d = np.array([math.cos(phi), math.sin(phi)])
        c = _centres(rng)
        f = _sources(n, n, 1.0, c)
        u = torch.zeros_like(f)
        for k in range(4):
            for cx, cy in c + 0.05 * k * d:
                u += 0.7 ** k * torch.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / (2.0 * (0.03 + 0.01 * k) ** 2))
        u /= u.max()
        cells = lambda g: g.reshape(HW, 4, HW, 4).permute(0, 2, 1, 3).reshape(HW, HW, 16)
        x[b, :, :, :16], x[b, :, :, 16:32] = cells(f), cells(u)
        x[b, :, :, 32], x[b, :, :, 33] = d[0], d[1]
        x[b, :, :, 34] = (rng.uniform(-4.0, -1.0) + 2.5) / 1.5
        x[b, :, :, 35], x[b, :, :, 36] = rng.uniform(-0.9, 1.0), 1.0
        t[b] = (rng.uniform(-0.2, 0.2) * cells(u).mean(-1)).float()
    return x.to(torch.bfloat16), t


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradient"):
        x, t = _net_inputs(case, seed)
        return dict(kind=kind, net=adr.Network(case["batch"], device=DEV), x=x, t=t)
    if kind == "batch":
        opts = dict(tol=case["tol"], max_iter=200000, prec=case["prec"], interp_weights=1,
                    anderson=case["anderson"])
        solvers = [adr.Solver(p, device=DEV, **opts) for p in _batch_problems(case, seed)]
        return dict(kind=kind, batch=adr.Batch(solvers))
    p = _problem(case, seed)
    st = dict(kind=kind, case=case, problem=p)
    if kind == "new":
        return st
    st["solver"] = adr.Solver(p, device=DEV, **_options(case))
    if kind == "split":
        g = torch.Generator(device="cpu").manual_seed(seed)
        u = torch.randn((p.ny, p.nx), dtype=torch.float64, generator=g).to(DEV)
        u[0, :] = u[-1, :] = 0.0
        u[:, 0] = u[:, -1] = 0.0
        st["u"] = u
        st["dt"] = 0.05
    elif p.u0 is not None:
        st["u"] = p.u0
    elif kind == "steps":  # the paper starts from its own u0
        st["u"] = st["solver"].paper_u0()
    return st


# -------------------------------------------------------------------- runs

def run(state):
    kind = state["kind"]
    if kind == "forward":
        return state["net"].forward(state["x"])
    if kind == "gradient":
        loss, grad = state["net"].loss_grad(state["x"], state["t"])
        return dict(loss=loss, grad=grad)
    if kind == "batch":
        outs, stats, _ = state["batch"].solve()
        return dict(u=outs, iters=np.array([s["iters"] for s in stats]))
    if kind == "split":
        half, nxt = state["solver"].split_step(state["u"], state["dt"])
        return dict(half=half, next=nxt)
    if kind == "new":
        s = adr.Solver(state["problem"], device=DEV, **_options(state["case"]))
        u, _, stats, _ = s.solve_stationary()
        s.close()
        return dict(u=u, iters=stats["iters"])
    if kind == "solve":
        u, _, stats, _ = state["solver"].solve_stationary()
        return dict(u=u, iters=stats["iters"])
    case = state["case"]
    u = state["u"].clone()
    stats, _ = state["solver"].step_parabolic(u, case["dt"], case["nsteps"], 1 if kind == "slices" else 0)
    return dict(u=u, iters=stats["iters"])


# -------------------------------------------------------------------- work

def _net_flops(batch):
    ch = W.CNN_CHANNELS
    return 2.0 * batch * HW * HW * sum(9 * a * b for a, b in zip(ch[:-1], ch[1:]))


def _steps(case, n):
    """Split steps of a solve, from the iteration's observed growth with the grid."""
    if case["kind"] in ("split", "steps"):
        return case.get("nsteps", 1)
    s = 60.0 + 12.0 * max(0.0, math.log2(n / 64.0))
    if case["kind"] == "slices":
        s *= 0.2 * case["nsteps"]
    return s


def work(case):
    """Bytes: each input field read once and each output written once.
    Operations: per split step and node of the grid about one unknown of each
    family, 7 + 14 + 16 operations for its sample, its solve and its map."""
    kind = case["kind"]
    if kind in ("forward", "gradient"):
        B, P = case["batch"], adr.adr_cnn_num_params()
        cells = B * HW * HW
        io = cells * 80.0 + (32.0 * cells if kind == "forward" else 4.0 * cells + 4.0 * P) + 4.0 * P
        return dict(bytes=io, flops=_net_flops(B) * (1.0 if kind == "forward" else 3.0))
    if kind == "batch":
        fixed = np.random.Generator(np.random.PCG64([W.SEED_BASE + 3, case["base"]]))
        b = fl = 0.0
        for _ in range(case["count"]):
            n = int(fixed.integers(case["nmin"], case["nmax"] + 1))
            kind_ = W.MASKS[int(fixed.integers(0, len(W.MASKS)))]
            fixed.uniform(size=3)
            nodes = n * n * {"square": 1.0, "disc": 0.636, "L": 0.75}[kind_]
            b += 33.0 * n * n
            fl += 74.0 * nodes * 2.0 * _steps(dict(kind="solve"), n)
        return dict(bytes=b, flops=fl)
    nodes = case["nx"] * case["ny"]
    per = {"split": 24.0, "steps": 16.0, "slices": 16.0}.get(kind, 33.0)
    return dict(bytes=per * nodes, flops=74.0 * nodes * _steps(case, max(case["nx"], case["ny"])))


# ------------------------------------------------------------------- exact

class _Lines:
    """One family of straight lines across a rectangle (constant slanted field)
    with its 1D systems, in the padded form [line][node]."""

    def __init__(self, p, fam, hs, hx, hy):
        bx, by = float(p.beta1[0, 0]), float(p.beta2[0, 0])
        nb = math.hypot(bx, by)
        bx, by = bx / nb, by / nb
        d = np.array([bx, by]) if fam == 0 else np.array([by, -bx])
        q = np.array([by, -bx]) if fam == 0 else np.array([bx, by])
        box = np.array([p.x1 - p.x0, p.y1 - p.y0])
        corners = [0.0, q[0] * box[0], q[1] * box[1], q @ box]
        ks = np.arange(math.ceil(min(corners) / hs - 1e-9), math.floor(max(corners) / hs + 1e-9) + 1)
        o = ks[:, None] * hs * q[None, :]
        lo, hi = -o / d, (box - o) / d
        sa, sb = np.minimum(lo, hi).max(1), np.maximum(lo, hi).min(1)
        keep = sb - sa > 1e-9 * hs
        self.k0, ks, o, sa, sb = int(ks[keep][0]), ks[keep], o[keep], sa[keep], sb[keep]
        self.sa, self.o, self.d, self.q = sa, o, d, q
        self.n = np.maximum(1, np.ceil((sb - sa) / hs - 1e-9)).astype(int)
        self.h = (sb - sa) / self.n
        j = np.arange(self.n.max() + 1)
        s = np.where(j[None, :] < self.n[:, None], sa[:, None] + j * self.h[:, None], sb[:, None])
        self.inner = (j[None, :] > 0) & (j[None, :] < self.n[:, None])
        self.xi = np.clip((o[:, :1] + s * d[0]) / hx, 0.0, p.nx - 1.0)
        self.eta = np.clip((o[:, 1:] + s * d[1]) / hy, 0.0, p.ny - 1.0)
        h = self.h[:, None]
        M, K = (h / 6.0, 2.0 * h / 3.0, h / 6.0), (-1.0 / h, 2.0 / h, -1.0 / h)
        C, sig = ((-0.5 * nb, 0.0, 0.5 * nb), p.sigma) if fam == 0 else ((0.0, 0.0, 0.0), 0.0)
        self.M = M
        self.S = tuple(p.mu * k + c + sig * m for k, c, m in zip(K, C, M))

    def sample(self, g):
        i = np.minimum(self.xi.astype(int), g.shape[1] - 2)
        r = np.minimum(self.eta.astype(int), g.shape[0] - 2)
        a, b = self.xi - i, self.eta - r
        return ((1 - a) * (1 - b) * g[r, i] + a * (1 - b) * g[r, i + 1] + (1 - a) * b * g[r + 1, i]
                + a * b * g[r + 1, i + 1])

    @staticmethod
    def _row(c, v):
        out = np.zeros_like(v)
        out[:, 1:-1] = c[0] * v[:, :-2] + c[1] * v[:, 1:-1] + c[2] * v[:, 2:]
        return out

    def substep(self, u, load, theta, dt):
        """v of (M + theta dt S) v = dt F + (M - (1 - theta) dt S) u, 0 at the ends."""
        u = np.where(self.inner, u, 0.0)
        r = self._row([m - (1 - theta) * dt * s for m, s in zip(self.M, self.S)], u)
        if load is not None:
            r = r + dt * self._row(self.M, load)
        a, b, c = (np.broadcast_to(m + theta * dt * s, (len(self.n), 1))[:, 0] for m, s in zip(self.M, self.S))
        J = u.shape[1]
        cp, rp = np.zeros_like(u), np.zeros_like(u)
        for j in range(1, J - 1):
            den = b - a * cp[:, j - 1]
            cp[:, j], rp[:, j] = np.where(self.inner[:, j], (c / den, (r[:, j] - a * rp[:, j - 1]) / den), 0.0)
        v = np.zeros_like(u)
        for j in range(J - 2, 0, -1):
            v[:, j] = np.where(self.inner[:, j], rp[:, j] - cp[:, j] * v[:, j + 1], 0.0)
        return v

    def crossings(self, nx, ny, hx, hy):
        """Per interior node and axis: the nearest lines before and after it on
        its row / column (flat node index, position in the element, weight)."""
        I, R = np.meshgrid(np.arange(1, nx - 1), np.arange(1, ny - 1))
        hs = min(hx, hy)
        out = []
        for ax, (pos, fix, hh) in enumerate(((I * hx, R * hy, hx), (R * hy, I * hx, hy))):
            qa, qb = self.q[ax], self.q[1 - ax]
            top = (nx - 1) * hx if ax == 0 else (ny - 1) * hy
            kk = (qa * pos + qb * fix) / hs
            kk = np.where(np.abs(kk - np.round(kk)) < 1e-9, np.round(kk), kk)
            below, above = (np.floor(kk), np.ceil(kk)) if qa > 0 else (np.ceil(kk), np.floor(kk))
            side = []
            for k, edge in ((below, 0.0), (above, top)):
                c = (k * hs - qb * fix) / qa
                ok = (c > 0.0) & (c < top) & (k >= self.k0) & (k < self.k0 + len(self.n))
                c = np.where(ok, c, edge)
                line = np.clip(k.astype(int) - self.k0, 0, len(self.n) - 1)
                pt = np.stack([c, fix] if ax == 0 else [fix, c], -1)
                s = (((pt - self.o[line]) @ self.d) - self.sa[line]) / self.h[line]
                j = np.clip(np.floor(s).astype(int), 0, self.n[line] - 1)
                side.append((ok, line, j, s - j, c))
            gap = side[1][4] - side[0][4]
            w = np.where(gap > 0.0, (pos - side[0][4]) / np.where(gap > 0.0, gap, 1.0), 0.0)
            out.append((side, w))
        self.cross = out

    def to_grid(self, v, nx, ny):
        g = np.zeros((ny, nx))
        for side, w in self.cross:
            val = [np.where(ok, (1 - t) * v[line, j] + t * v[line, j + 1], 0.0) for ok, line, j, t, _ in side]
            g[1:-1, 1:-1] += 0.5 * ((1 - w) * val[0] + w * val[1])
        return g


def _exact_slant(case, seed):
    """The split scheme of a constant slanted field on a rectangle, in plain
    numpy: the same discretisation, serial elimination line by line."""
    p = _problem(case, seed)
    nx, ny = p.nx, p.ny
    hx, hy = (p.x1 - p.x0) / (nx - 1), (p.y1 - p.y0) / (ny - 1)
    hs = min(hx, hy)
    B, G = (_Lines(p, fam, hs, hx, hy) for fam in (0, 1))
    for L in (B, G):
        L.crossings(nx, ny, hx, hy)
    load = B.sample(p.f.cpu().numpy())

    def step(u, dt):
        half = B.to_grid(B.substep(B.sample(u), load, 0.5, dt), nx, ny)
        return half, G.to_grid(G.substep(G.sample(half), None, 0.5, dt), nx, ny)

    if case["kind"] == "split":
        st = torch.Generator(device="cpu").manual_seed(seed)
        u = torch.randn((ny, nx), dtype=torch.float64, generator=st).numpy()
        u[0, :] = u[-1, :] = 0.0
        u[:, 0] = u[:, -1] = 0.0
        half, nxt = step(u, 0.05)
        return dict(half=half, next=nxt)
    bmax = math.hypot(float(p.beta1[0, 0]), float(p.beta2[0, 0]))
    dt = 2.0 / math.sqrt(p.sigma * (12.0 * p.mu / hs ** 2 + 2.0 * math.sqrt(3.0) * bmax / hs))
    u, k = np.zeros((ny, nx)), 0
    while k < 100000:
        half, nxt = step(u, dt)
        k += 1
        rel = math.sqrt(((nxt - u) ** 2).sum() / (nxt ** 2).sum())
        mid, u = 0.5 * (u + half), nxt
        if rel <= case["tol"]:
            break
    return dict(u=mid, iters=k)


def _exact_net(case, seed):
    """The network in FP64 on the same features and targets (cuDNN's or
    PyTorch's own 64-bit convolutions, a few problems at a time)."""
    xs, ts = _net_inputs(case, seed)
    params = torch.as_tensor(W.cnn_init_params(), device=DEV).double()
    dil, ch = (1, 2, 4, 8, 16, 32, 1, 1), W.CNN_CHANNELS
    layers, off = [], 0
    for a, b in zip(ch[:-1], ch[1:]):
        layers.append((off, off + 9 * a * b, off + 9 * a * b + b, a, b))
        off += 9 * a * b + b
    train = case["kind"] == "gradient"
    params.requires_grad_(train)
    cells = float(case["batch"] * HW * HW)
    outs, loss = [], 0.0
    for k in range(0, case["batch"], 8):
        h = xs[k:k + 8].double().permute(0, 3, 1, 2)
        for l, (o, ob, oe, a, b) in enumerate(layers):
            w = params[o:ob].reshape(3, 3, a, b).permute(3, 2, 0, 1)
            h = torch.nn.functional.conv2d(h, w, params[ob:oe], padding=dil[l], dilation=dil[l])
            if l + 1 < len(layers):
                h = torch.relu(h)
        if train:
            e = 0.5 * ((h[:, 0] - ts[k:k + 8].double()) ** 2).sum() / cells
            e.backward()
            loss += float(e)
        else:
            outs.append(h.permute(0, 2, 3, 1).contiguous())
    return dict(loss=loss, grad=params.grad) if train else torch.cat(outs)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("forward", "gradient"):
        return _exact_net(case, seed)
    if case.get("field") == "slant" and kind in ("split", "solve"):
        small = case["nx"] * case["ny"] <= (700 * 700 if kind == "split" else 250 * 250)
        if small and not (case.get("prec") or case.get("transfer") or case.get("anderson")):
            return _exact_slant(case, seed)
    return None  # traced curves, masked domains, large solves: minutes in plain numpy
