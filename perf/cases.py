"""The performance cases of the library: what its users have it compute, each
through the public calls of ``paper_1111_6583_gb300.claw``.

A case is one grid (``Solver.evolve`` for a number of steps, as a program
advances to its next output frame), an ensemble of uneven grids (``Batch``) or
a stream of requests (``Server``), with Clawpack-classic or SharpClaw, in FP64
or FP32.  ``exact`` restates the methods in plain FP64 torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

FAR = 1e30  # a final time that no case reaches


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # the 1D acoustics line of the paper's examples: a small grid, many
        # steps, where the latency of a step counts
        dict(name="line_2000_fp64", kind="line", prec="fp64", nx=2000, steps=160, lim="mc"),
        # a long line in FP32: the streaming end of the same path
        dict(name="line_2p25_fp32", kind="line", prec="fp32", nx=1 << 25, steps=16, lim="mc"),
        # nonlinear elasticity in layered media: many uneven 1D grids at once
        dict(name="ensemble_256_fp32", kind="ensemble", prec="fp32", members=256, lo=12, hi=16,
             mix=1, steps=64),
        # the radial dam break with a Roe solver and transverse terms, plain FP64
        dict(name="dambreak_1024_fp64", kind="dambreak", prec="fp64", nx=1024, ny=1024, steps=16,
             lim="mc"),
        # the same in FP32 on the largest grid a single run uses
        dict(name="dambreak_4096_fp32", kind="dambreak", prec="fp32", nx=4096, ny=4096, steps=16,
             lim="mc"),
        # a service: requests of mixed sizes and final times from host memory
        dict(name="serve_24_fp32", kind="serve", prec="fp32", requests=24, lo=64, hi=384, mix=2),
        # 2D constant-medium acoustics on a ragged grid, FP64
        dict(name="acoustics2d_1000_fp64", kind="acoustics2d", prec="fp64", nx=1000, ny=750,
             steps=16, lim="mc"),
        # 3D acoustics with transverse and double-transverse terms, FP32
        dict(name="acoustics3d_256_fp32", kind="acoustics3d", prec="fp32", nx=256, ny=256, nz=256,
             steps=16, lim="mc"),
        # shock-bubble interaction, SharpClaw WENO5 + SSP-RK3, FP64 plain form
        dict(name="bubble_2048_fp64", kind="bubble", prec="fp64", nx=2048, ny=1024, steps=4),
        # the same in FP32 on a ragged grid
        dict(name="bubble_1500_fp32", kind="bubble", prec="fp32", nx=1500, ny=700, steps=16),
        # axisymmetric shock-bubble: Euler with a tracer and a geometric source
        dict(name="axisym_1280_fp64", kind="axisym", prec="fp64", nx=1280, ny=320, steps=16,
             lim="mc", split="godunov"),
        # acoustics in a varying medium on a stretched grid (capacity form)
        dict(name="medium_1024_fp32", kind="medium", prec="fp32", nx=1024, ny=1024, steps=16,
             lim="mc", capacity=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["line", "ensemble", "dambreak", "serve", "acoustics2d", "acoustics3d",
                       "bubble", "axisym", "medium"])
    prec = rng.choice(["fp32", "fp64"])
    f64 = prec == "fp64"
    lim = rng.choice(["mc", "mc", "mc", "superbee", "minmod", "vanleer"])
    if kind == "line":
        n = _log(rng, 500, (1 << 22) if f64 else (1 << 25))
        return dict(kind=kind, prec=prec, nx=n, steps=160 if n < 100000 else 16, lim=lim)
    if kind == "ensemble":
        return dict(kind=kind, prec=prec, members=_log(rng, 16, 48 if f64 else 256), lo=12,
                    hi=rng.choice([13, 14, 15, 16]), mix=rng.randrange(1000), steps=64)
    if kind == "serve":
        return dict(kind=kind, prec=prec, requests=rng.randint(8, 24), lo=64,
                    hi=rng.choice([96, 128, 160]) if f64 else rng.choice([128, 256, 384]),
                    mix=rng.randrange(1000))
    if kind == "acoustics3d":
        n = _log(rng, 24, 144 if f64 else 256)
        a, b, c = (max(16, min(256, int(round(n * rng.uniform(0.7, 1.3))))) for _ in range(3))
        return dict(kind=kind, prec=prec, nx=a, ny=b, nz=c, steps=16, lim=lim)
    if kind == "bubble":
        nx = _log(rng, 128, 1024 if f64 else 2048)
        return dict(kind=kind, prec=prec, nx=nx, ny=int(nx * rng.uniform(0.4, 0.6)),
                    steps=4 if f64 else 16)
    if kind == "axisym":
        nx = _log(rng, 160, 1280)
        return dict(kind=kind, prec=prec, nx=nx, ny=int(nx * rng.uniform(0.2, 0.3)), steps=16,
                    lim=lim, split=rng.choice(["godunov", "strang"]))
    if kind == "medium":
        n = _log(rng, 64, 1024)
        return dict(kind=kind, prec=prec, nx=n, ny=int(n * rng.uniform(0.8, 1.0)), steps=16,
                    lim=lim, capacity=rng.random() < 0.5)
    n = _log(rng, 64, 1024 if f64 else 4096)  # dambreak, acoustics2d
    return dict(kind=kind, prec=prec, nx=n, ny=int(n * rng.uniform(0.7, 1.0)), steps=16, lim=lim)


def _cells(case):
    return case["nx"] * case.get("ny", 1) * case.get("nz", 1)


# per cell and step: fields of the state, fields of aux, floating-point
# operations of the method (solves, limited corrections, transverse terms)
_PER_CELL = {"line": (2, 0, 60), "ensemble": (2, 2, 96), "dambreak": (3, 0, 825),
             "serve": (3, 0, 825), "acoustics2d": (3, 0, 120), "acoustics3d": (4, 0, 260),
             "bubble": (4, 0, 3 * 2400), "axisym": (5, 0, 1000), "medium": (3, 2, 260)}


def work(case):
    """Each step reads the state (and aux) once and writes it once: the next
    step's dt depends on every cell of this one."""
    m, ma, fl = _PER_CELL[case["kind"]]
    if case["kind"] == "medium" and case["capacity"]:
        ma = 3
    es = 8 if case["prec"] == "fp64" else 4
    if case["kind"] == "ensemble":
        cs = sum(_ensemble_sizes(case)) * case["steps"]
    elif case["kind"] == "serve":
        # about 1.6 cells per unit of time and cell width at Courant number 0.9
        cs = sum(n * n * math.ceil(1.6 * t * n / 0.9) for n, t in _serve_mix(case))
    else:
        cs = _cells(case) * case["steps"]
    return {"bytes": cs * es * (2 * m + ma), "flops": cs * fl}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _ensemble_sizes(case):
    r = random.Random(case["mix"])
    return [round(2.0 ** (case["lo"] + (case["hi"] - case["lo"]) * r.random()))
            for _ in range(case["members"])]


def _serve_mix(case):
    r = random.Random(case["mix"])
    return [(round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"])))),
             r.uniform(0.05, 0.15)) for _ in range(case["requests"])]


def _centers(lo, hi, n):
    return lo + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * ((hi - lo) / n)


def _base(ndim, n, lower, upper, rp, **kw):
    spec = dict(ndim=ndim, n=list(n), lower=list(lower), upper=list(upper), rp=rp,
                scheme="classic", lim="mc", order=2, transverse=2, char_decomp=0, entropy_fix=1,
                weno_eps=1e-6, bc_lower=["periodic"] * ndim, bc_upper=["periodic"] * ndim,
                inflow=[], params=[], cfl_desired=0.9, cfl_max=1.0, dt_initial=0.0, dt_max=1e30,
                max_retries=8)
    spec.update(kw)
    return spec


def _inside(X, Y, dx, dy, cx, cy, r, sub=4):
    """Fraction of each cell inside a disc, from sub x sub sample points."""
    f = torch.zeros(torch.broadcast_shapes(X.shape, Y.shape), dtype=torch.float64, device="cuda")
    for a in range(sub):
        for b in range(sub):
            xs = X + ((a + 0.5) / sub - 0.5) * dx
            ys = Y + ((b + 0.5) / sub - 0.5) * dy
            f += ((xs - cx) ** 2 + (ys - cy) ** 2 < r * r)
    return f / (sub * sub)


def _post_shock(p2, gamma=1.4):
    """Rankine-Hugoniot state behind a shock into rho = p = 1 at rest."""
    m2 = 1.0 + (gamma + 1.0) / (2.0 * gamma) * (p2 - 1.0)
    rho2 = (gamma + 1.0) * m2 / ((gamma - 1.0) * m2 + 2.0)
    return rho2, math.sqrt(m2 * gamma) * (1.0 - 1.0 / rho2)


def _grid_inputs(case, seed):
    """(spec, q0, aux) of a single-grid case; q0, aux FP64 on the GPU."""
    r = random.Random(seed)
    kind = case["kind"]
    aux = None
    if kind == "line":
        x = _centers(-1.0, 1.0, case["nx"])
        c, a = r.uniform(-0.3, 0.0), r.uniform(0.8, 1.2)
        p = torch.exp(-100.0 * (x - c) ** 2) + a * ((x >= 0.3) & (x <= 0.5))
        q0 = torch.stack([p, torch.zeros_like(p)])
        spec = _base(1, [case["nx"]], [-1.0], [1.0], "acoustics", params=[1.0, 4.0])
    elif kind in ("acoustics2d", "acoustics3d"):
        nd = 2 if kind == "acoustics2d" else 3
        n = [case["nx"], case["ny"], case.get("nz", 1)][:nd]
        up = [n[d] / n[0] for d in range(nd)]  # square cells on [-a, a]^d
        xs = [_centers(-u, u, m) for u, m in zip(up, n)]
        r2, box = 0.0, True
        for d in range(nd):
            v = xs[d].reshape([-1] + [1] * d)
            r2 = r2 + (v - r.uniform(-0.1, 0.1)) ** 2
            box = box & (v >= 0.3 * up[d]) & (v <= 0.5 * up[d])
        p = torch.exp(-100.0 * r2) + r.uniform(0.8, 1.2) * box
        q0 = torch.stack([p] + [torch.zeros_like(p)] * nd)
        spec = _base(nd, n, [-u for u in up], up, "acoustics", params=[1.0, 4.0],
                     bc_lower=["wall"] * nd, bc_upper=["wall"] * nd)
    elif kind == "dambreak":
        asp = case["ny"] / case["nx"]
        x = _centers(-2.5, 2.5, case["nx"])
        y = _centers(-2.5 * asp, 2.5 * asp, case["ny"])[:, None]
        rad, cx, cy = r.uniform(0.45, 0.55), r.uniform(-0.2, 0.2), r.uniform(-0.2, 0.2)
        h = torch.where((x - cx) ** 2 + (y - cy) ** 2 < rad * rad, r.uniform(1.8, 2.2), 1.0)
        h = h.to(torch.float64)
        q0 = torch.stack([h, torch.zeros_like(h), torch.zeros_like(h)])
        spec = _base(2, [case["nx"], case["ny"]], [-2.5, -2.5 * asp], [2.5, 2.5 * asp], "sw_roe",
                     params=[1.0], bc_lower=["wall", "wall"], bc_upper=["wall", "wall"])
    elif kind in ("bubble", "axisym"):
        g = 1.4
        top = 1.0 if kind == "bubble" else 0.5
        x = _centers(0.0, 2.0, case["nx"])
        y = _centers(0.0, top, case["ny"])[:, None]
        cy = 0.5 + r.uniform(-0.05, 0.05) if kind == "bubble" else 0.0
        f = _inside(x, y, 2.0 / case["nx"], top / case["ny"], 0.5 + r.uniform(-0.05, 0.05), cy,
                    r.uniform(0.18, 0.22))
        rho2, u2 = _post_shock(4.5 if kind == "bubble" else 5.0, g)
        p2 = 4.5 if kind == "bubble" else 5.0
        E2 = p2 / (g - 1.0) + 0.5 * rho2 * u2 * u2
        left = (x < 0.2) & (y > -1.0)
        rho = torch.where(left, rho2, f * r.uniform(0.1, 0.2) + (1.0 - f))
        z = torch.zeros_like(rho)
        q = [rho, torch.where(left, rho2 * u2, 0.0).to(torch.float64), z,
             torch.where(left, E2, 1.0 / (g - 1.0)).to(torch.float64)]
        if kind == "bubble":
            spec = _base(2, [case["nx"], case["ny"]], [0.0, 0.0], [2.0, 1.0], "euler_roe",
                         scheme="sharpclaw", char_decomp=1, params=[g],
                         bc_lower=["inflow", "wall"], bc_upper=["extrap", "wall"],
                         inflow=[rho2, rho2 * u2, 0.0, E2], cfl_desired=0.5, cfl_max=0.6)
        else:
            q.append(torch.where(left, 0.0, f))
            spec = _base(2, [case["nx"], case["ny"]], [0.0, 0.0], [2.0, 0.5], "euler_tracer",
                         params=[g], source="axisymmetric", source_split=case["split"],
                         bc_lower=["inflow", "wall"], bc_upper=["extrap", "extrap"],
                         inflow=[rho2, rho2 * u2, 0.0, E2, 0.0], cfl_desired=0.8)
        q0 = torch.stack(q)
    elif kind == "medium":
        asp = case["ny"] / case["nx"]
        xi = _centers(-1.0, 1.0, case["nx"])
        y = _centers(-asp, asp, case["ny"])[:, None]
        x = xi + 0.1 * torch.sin(math.pi * xi) if case["capacity"] else xi
        one = torch.ones_like(xi * y)
        xm = 0.3 + r.uniform(-0.1, 0.1)
        a = [torch.where(x < xm, 1.0, 4.0) * one, torch.where(x < xm, 1.0, 0.5) * one]
        kw = {}
        if case["capacity"]:
            a.append((1.0 + 0.1 * math.pi * torch.cos(math.pi * xi)) * one)
            kw["capa_index"] = 2
        aux = torch.stack(a)
        p = torch.exp(-80.0 * ((x + 0.4 + r.uniform(-0.1, 0.1)) ** 2 + y ** 2))
        q0 = torch.stack([p, torch.zeros_like(p), torch.zeros_like(p)])
        spec = _base(2, [case["nx"], case["ny"]], [-1.0, -asp], [1.0, asp], "acoustics_vc",
                     num_aux=len(a), bc_lower=["wall", "wall"], bc_upper=["wall", "wall"], **kw)
    else:
        raise ValueError(kind)
    spec["lim"] = case.get("lim", "mc")
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    return spec, q0.to(dt).contiguous(), aux.to(dt).contiguous() if aux is not None else None


def _ensemble_inputs(case, seed):
    """The members' specs; their states and media are views of two flat
    buffers, each member's on a 512-byte boundary like an allocation's."""
    r = random.Random(seed)
    dt = torch.float64 if case["prec"] == "fp64" else torch.float32
    sizes = _ensemble_sizes(case)
    pad = [-(-2 * n // 128) * 128 for n in sizes]
    flat, med = (torch.zeros(sum(pad), dtype=dt, device="cuda") for _ in range(2))
    specs, at = [], 0
    dx = 1.0 / 32.0
    for n, w in zip(sizes, pad):
        x = _centers(0.0, n * dx, n)
        odd = torch.floor(x / 0.5).to(torch.int64) % 2 == 1
        m = torch.where(odd, 4.0, 1.0).to(torch.float64)
        amp, width = r.uniform(0.1, 0.5), r.uniform(1.0, 5.0)
        sig = amp * torch.exp(-((x - 0.5 * n * dx) / width) ** 2)
        q = flat[at:at + 2 * n].view(2, n)
        a = med[at:at + 2 * n].view(2, n)
        q[0] = (torch.log1p(sig) / m).to(dt)
        a[:] = m.to(dt)
        spec = _base(1, [n], [0.0], [n * dx], "elasticity_fwave", num_aux=2)
        spec.update(q0=q, aux=a, t_end=FAR)
        specs.append(spec)
        at += w
    return specs, flat


def _serve_inputs(case, seed):
    """The requests' specs, initial states in host memory."""
    r = random.Random(seed)
    dt = np.float64 if case["prec"] == "fp64" else np.float32
    specs = []
    for n, t_end in _serve_mix(case):
        x = (np.arange(n) + 0.5) / n
        h = np.ones((n, n))
        for _ in range(r.randint(1, 3)):
            a, w = r.uniform(0.1, 1.0), r.uniform(0.05, 0.3)
            cx, cy = r.uniform(0.15, 0.85), r.uniform(0.15, 0.85)
            h += a * np.exp(-((x[:, None] - cy) / w) ** 2) * np.exp(-((x - cx) / w) ** 2)
        q0 = np.zeros((3, n, n), dtype=dt)
        q0[0] = h
        spec = _base(2, [n, n], [0.0, 0.0], [1.0, 1.0], "sw_roe", params=[1.0],
                     bc_lower=["wall", "wall"], bc_upper=["wall", "wall"])
        spec.update(q0=q0, aux=None, t_end=t_end)
        specs.append(spec)
    return specs


def prepare(case, seed):
    from paper_1111_6583_gb300 import claw

    if case["kind"] == "ensemble":
        specs, flat = _ensemble_inputs(case, seed)
        return dict(case=case, batch=claw.Batch(specs, case["prec"]), flat=flat)
    if case["kind"] == "serve":
        specs = _serve_inputs(case, seed)
        return dict(case=case, specs=specs, server=claw.Server(specs[0], case["prec"]))
    spec, q0, aux = _grid_inputs(case, seed)
    q = q0.clone()
    return dict(case=case, q0=q0, q=q, solver=claw.Solver(spec, case["prec"], q=q, aux=aux))


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        # carry every member on by that many steps
        state["batch"].advance(case["steps"])
        state["batch"].sync()
        return state["flat"]
    if case["kind"] == "serve":
        server = state["server"]
        tickets = [server.submit(s) for s in state["specs"]]
        while True:
            running, queued = server.pump(8)
            if not running and not queued:
                break
        return [server.poll(t)["q"] for t in tickets]
    # the program writes the state to start from into the solver's buffer and
    # advances it to the next frame
    state["q"].copy_(state["q0"])
    info = state["solver"].evolve(FAR, max_steps=case["steps"])
    return {"q": state["q"], "steps": info["steps"], "rejects": info["rejects"]}


# --------------------------------------------------------------------------
# the methods in plain FP64 torch.  Arrays are [field][nz][ny][nx] with ghost
# cells; face i of direction d lies between cells i - 1 and i.
# --------------------------------------------------------------------------
def _roll(x, k, d):
    return torch.roll(x, k, -1 - d)


def _ghosts(q, g, spec, aux=False):
    """Ghost cells direction by direction (x, then y on the result, then z)."""
    for d in range(spec["ndim"]):
        ax, n = q.dim() - 1 - d, q.shape[-1 - d]
        parts = []
        for side, bc in ((0, spec["bc_lower"][d]), (1, spec["bc_upper"][d])):
            if bc == "periodic":
                p = q.narrow(ax, n - g, g) if side == 0 else q.narrow(ax, 0, g)
            elif bc == "wall":
                p = (q.narrow(ax, 0, g) if side == 0 else q.narrow(ax, n - g, g)).flip(ax)
                if not aux:
                    p = p.clone()
                    p[1 + d] = -p[1 + d]
            else:
                p = q.narrow(ax, 0 if side == 0 else n - 1, 1)
                p = p.expand([g if a == ax else s for a, s in enumerate(p.shape)])
                if bc == "inflow" and not aux:
                    v = torch.tensor(spec["inflow"][:q.shape[0]], dtype=q.dtype, device=q.device)
                    p = v.reshape([-1] + [1] * (q.dim() - 1)).expand(p.shape)
            parts.append(p)
        q = torch.cat([parts[0], q, parts[1]], dim=ax)
    return q


def _phi(lim, th):
    if lim == "minmod":
        return th.clamp(0.0, 1.0)
    if lim == "superbee":
        return torch.maximum(torch.minimum(torch.ones_like(th), 2 * th),
                             torch.minimum(torch.full_like(th, 2.0), th)).clamp(min=0.0)
    if lim == "vanleer":
        return (th + th.abs()) / (1.0 + th.abs())
    return torch.minimum(0.5 * (1.0 + th), 2.0 * th).clamp(0.0, 2.0)


class _Acoustics:
    fwave = False

    def __init__(self, spec):
        rho, K = spec["params"][:2]
        self.c = math.sqrt(K / rho)
        self.Z = rho * self.c

    def solve(self, d, ql, qr, al, ar):
        n, Z, c = 1 + d, self.Z, self.c
        dp, du = qr[0] - ql[0], qr[n] - ql[n]
        one = torch.ones_like(dp)
        W = [torch.zeros_like(ql), torch.zeros_like(ql)]
        a1, a2 = (Z * du - dp) / (2 * Z), (Z * du + dp) / (2 * Z)
        W[0][0], W[0][n] = -Z * a1, a1
        W[1][0], W[1][n] = Z * a2, a2
        return W, [-c * one, c * one], -c * W[0], c * W[1], None

    def split(self, e, a):
        n, Z, c = 1 + e, self.Z, self.c
        b1, b2 = (Z * a[n] - a[0]) / (2 * Z), (Z * a[n] + a[0]) / (2 * Z)
        em, ep = torch.zeros_like(a), torch.zeros_like(a)
        em[0], em[n] = c * Z * b1, -c * b1
        ep[0], ep[n] = c * Z * b2, c * b2
        return em, ep

    def trans(self, d, ctx, a, aux):
        return self.split(1 - d, a)


class _Medium:
    fwave = False

    def solve(self, d, ql, qr, al, ar):
        n = 1 + d
        Zl, Zr = al[0] * al[1], ar[0] * ar[1]
        dp, du = qr[0] - ql[0], qr[n] - ql[n]
        a1, a2 = (Zr * du - dp) / (Zl + Zr), (Zl * du + dp) / (Zl + Zr)
        W = [torch.zeros_like(ql), torch.zeros_like(ql)]
        W[0][0], W[0][n] = -a1 * Zl, a1
        W[1][0], W[1][n] = a2 * Zr, a2
        return W, [-al[1], ar[1]], -al[1] * W[0], ar[1] * W[1], None

    def trans(self, d, ctx, a, aux):
        e, n = 1 - d, 2 - d
        lo, hi = _roll(aux, 1, e), _roll(aux, -1, e)
        Zm, Zc, Zp = lo[0] * lo[1], aux[0] * aux[1], hi[0] * hi[1]
        b1, b2 = (Zc * a[n] - a[0]) / (Zm + Zc), (Zc * a[n] + a[0]) / (Zc + Zp)
        bm, bp = torch.zeros_like(a), torch.zeros_like(a)
        bm[0], bm[n] = lo[1] * b1 * Zm, -lo[1] * b1
        bp[0], bp[n] = hi[1] * b2 * Zp, hi[1] * b2
        return bm, bp


class _Elasticity:
    fwave = True

    def solve(self, d, ql, qr, al, ar):
        el, er = torch.exp(al[1] * ql[0]), torch.exp(ar[1] * qr[0])
        cl, cr = torch.sqrt(al[1] * el / al[0]), torch.sqrt(ar[1] * er / ar[0])
        Zl, Zr = al[0] * cl, ar[0] * cr
        d1, d2 = ql[1] / al[0] - qr[1] / ar[0], el - er
        b1, b2 = (Zr * d1 + d2) / (Zl + Zr), (Zl * d1 - d2) / (Zl + Zr)
        W = [torch.stack([b1, b1 * Zl]), torch.stack([b2, -b2 * Zr])]
        return W, [-cl, cr], W[0], W[1], None


def _harten_hyman(speed, ql, qr, W, s, am, ap):
    """Entropy fix of the first and last families (first one first)."""
    tot = sum(si * Wi for si, Wi in zip(s, W))
    qm = ql + W[0]
    l0, l1 = speed(ql, -1), speed(qm, -1)
    fix1 = (l0 < 0) & (l1 > 0)
    beta = (l1 - s[0]) / torch.where(fix1, l1 - l0, 1.0)
    am1 = beta * l0 * W[0]
    qm = qr - W[-1]
    r0, r1 = speed(qm, 1), speed(qr, 1)
    fix2 = (r0 < 0) & (r1 > 0) & ~fix1
    beta = (r1 - s[-1]) / torch.where(fix2, r1 - r0, 1.0)
    ap2 = (1.0 - beta) * r1 * W[-1]
    am, ap = torch.where(fix2, tot - ap2, am), torch.where(fix2, ap2, ap)
    return torch.where(fix1, am1, am), torch.where(fix1, tot - am1, ap)


def _by_speed(W, s):
    return (sum(torch.clamp(si, max=0.0) * Wi for si, Wi in zip(s, W)),
            sum(torch.clamp(si, min=0.0) * Wi for si, Wi in zip(s, W)))


class _ShallowWater:
    fwave = False

    def __init__(self, spec):
        self.g = spec["params"][0]

    @staticmethod
    def coef(un, ut, c, dh, dn, dt):
        return (((un + c) * dh - dn) / (2 * c), dt - ut * dh, (dn - (un - c) * dh) / (2 * c))

    def solve(self, d, ql, qr, al, ar):
        n, t = 1 + d, 2 - d
        sl, sr = torch.sqrt(ql[0]), torch.sqrt(qr[0])
        un = (ql[n] / sl + qr[n] / sr) / (sl + sr)
        ut = (ql[t] / sl + qr[t] / sr) / (sl + sr)
        c = torch.sqrt(self.g * 0.5 * (ql[0] + qr[0]))
        a0, a1, a2 = self.coef(un, ut, c, qr[0] - ql[0], qr[n] - ql[n], qr[t] - ql[t])
        W = [torch.zeros_like(ql) for _ in range(3)]
        W[0][0], W[0][n], W[0][t] = a0, a0 * (un - c), a0 * ut
        W[1][t] = a1
        W[2][0], W[2][n], W[2][t] = a2, a2 * (un + c), a2 * ut
        s = [un - c, un, un + c]
        am, ap = _by_speed(W, s)

        def speed(q, sg):
            return q[n] / q[0] + sg * torch.sqrt(self.g * q[0])

        am, ap = _harten_hyman(speed, ql, qr, W, s, am, ap)
        return W, s, am, ap, torch.stack([un, ut, c])

    def trans(self, d, ctx, a, aux):
        n, t = 1 + d, 2 - d
        un, ut, c = ctx
        b = self.coef(ut, un, c, a[0], a[t], a[n])
        lam = [ut - c, ut, ut + c]
        out = []
        for f in (lambda x: torch.clamp(x, max=0.0), lambda x: torch.clamp(x, min=0.0)):
            k = [f(li) * bi for li, bi in zip(lam, b)]
            o = torch.empty_like(a)
            o[0] = k[0] + k[2]
            o[t] = k[0] * lam[0] + k[2] * lam[2]
            o[n] = (k[0] + k[2]) * un + k[1]
            out.append(o)
        return out


class _Euler:
    """Euler (rho, m_x, m_y, E), optionally with an advected tracer."""
    fwave = False

    def __init__(self, spec, tracer=False):
        self.gm = spec["params"][0]
        self.tracer = tracer

    def pressure(self, q):
        return (self.gm - 1.0) * (q[3] - 0.5 * (q[1] ** 2 + q[2] ** 2) / q[0])

    def roe(self, d, ql, qr):
        n, t = 1 + d, 2 - d
        sl, sr = torch.sqrt(ql[0]), torch.sqrt(qr[0])
        un = (ql[n] / sl + qr[n] / sr) / (sl + sr)
        ut = (ql[t] / sl + qr[t] / sr) / (sl + sr)
        H = ((ql[3] + self.pressure(ql)) / sl + (qr[3] + self.pressure(qr)) / sr) / (sl + sr)
        c = torch.sqrt((self.gm - 1.0) * (H - 0.5 * (un * un + ut * ut)))
        return torch.stack([un, ut, H, c])

    def coef(self, un, ut, H, c, d0, dn, dt, dE):
        a2 = dt - ut * d0
        a1 = (self.gm - 1.0) * ((H - un * un) * d0 + un * dn - dE + ut * a2) / (c * c)
        a3 = (dn + (c - un) * d0 - c * a1) / (2 * c)
        return d0 - a1 - a3, a1, a2, a3

    @staticmethod
    def assemble(un, ut, H, c, k, n, t, like):
        o = torch.zeros_like(like)
        o[0] = k[0] + k[1] + k[3]
        o[n] = k[0] * (un - c) + k[1] * un + k[3] * (un + c)
        o[t] = (k[0] + k[1] + k[3]) * ut + k[2]
        o[3] = (k[0] * (H - un * c) + k[1] * 0.5 * (un * un + ut * ut) + k[2] * ut +
                k[3] * (H + un * c))
        return o

    def solve(self, d, ql, qr, al, ar):
        n, t = 1 + d, 2 - d
        un, ut, H, c = x = self.roe(d, ql, qr)
        D = qr - ql
        a = self.coef(un, ut, H, c, D[0], D[n], D[t], D[3])
        z = torch.zeros_like(un)
        W = [self.assemble(un, ut, H, c, [a[i] if i == p else z for i in range(4)], n, t, ql)
             for p in range(4)]
        s = [un - c, un, un, un + c]
        am, ap = _by_speed(W, s)

        def speed(q, sg):
            return q[n] / q[0] + sg * torch.sqrt(self.gm * self.pressure(q) / q[0])

        am, ap = _harten_hyman(speed, ql, qr, W, s, am, ap)
        if self.tracer:
            w = torch.zeros_like(ql)
            w[4] = D[4]
            W.append(w)
            s.append(un)
            am, ap = am + torch.clamp(un, max=0.0) * w, ap + torch.clamp(un, min=0.0) * w
        return W, s, am, ap, x

    def trans(self, d, ctx, a, aux):
        n, t = 1 + d, 2 - d
        un, ut, H, c = ctx
        b = self.coef(ut, un, H, c, a[0], a[t], a[n], a[3])
        out = []
        for f in (lambda x: torch.clamp(x, max=0.0), lambda x: torch.clamp(x, min=0.0)):
            k = [f(ut - c) * b[0], f(ut) * b[1], f(ut) * b[2], f(ut + c) * b[3]]
            o = self.assemble(ut, un, H, c, k, t, n, a)
            if self.tracer:
                o[4] = f(ut) * a[4]
            out.append(o)
        return out

    def flux(self, d, q):
        n, t = 1 + d, 2 - d
        u, p, f = q[n] / q[0], self.pressure(q), torch.empty_like(q)
        f[0], f[n], f[t], f[3] = q[n], q[n] * u + p, q[t] * u, u * (q[3] + p)
        return f


def _system(spec):
    return {"acoustics": _Acoustics, "sw_roe": _ShallowWater, "euler_roe": _Euler,
            "euler_tracer": lambda s: _Euler(s, True), "elasticity_fwave": lambda s: _Elasticity(),
            "acoustics_vc": lambda s: _Medium()}[spec["rp"]](spec)


def _dx(spec):
    return [(spec["upper"][d] - spec["lower"][d]) / spec["n"][d] for d in range(spec["ndim"])]


def _inner(x, nd, g):
    for d in range(nd):
        x = x.narrow(x.dim() - 1 - d, g, x.shape[-1 - d] - 2 * g)
    return x


def _face_speed(s, kap, d, nd):
    """Largest speed over the faces 0 .. n of interior lines."""
    best = 0.0
    for si in s:
        a = si.abs()
        if kap is not None:
            a = torch.where(si > 0, si / kap, -si / _roll(kap, 1, d))
        for e in range(nd):
            ax = a.dim() - 1 - e
            a = a.narrow(ax, 2, a.shape[ax] - 4 + (1 if e == d else 0))
        best = max(best, float(a.max()))
    return best


def _classic_step(S, spec, q, aux, dt):
    """(new state, per-direction largest speeds) of one unsplit step."""
    nd, lim = spec["ndim"], spec["lim"]
    lam = [dt / h for h in _dx(spec)]
    Q = _ghosts(q, 2, spec)
    A = _ghosts(aux, 2, spec, aux=True) if aux is not None else None
    kap = A[spec["capa_index"]] if spec.get("capa_index", -1) >= 0 else None
    out, speeds = Q.clone(), []
    ik = 1.0 if kap is None else 1.0 / kap
    for d in range(nd):
        Al = _roll(A, 1, d) if A is not None else None
        W, s, am, ap, ctx = S.solve(d, _roll(Q, 1, d), Q, Al, A)
        speeds.append(_face_speed(s, kap, d, nd))
        dtc = lam[d] if kap is None else 0.5 * lam[d] * (ik + _roll(ik, 1, d))
        F = torch.zeros_like(am)
        for Wp, sp in zip(W, s):
            up = torch.where(sp > 0, _roll(Wp, 1, d), _roll(Wp, -1, d))
            nrm = (Wp * Wp).sum(0)
            th = (up * Wp).sum(0) / torch.where(nrm == 0, 1.0, nrm)
            ph = torch.where(nrm == 0, 0.0, _phi(lim, th))
            a = sp.abs()
            F = F + 0.5 * (torch.sign(sp) if S.fwave else a) * (1.0 - dtc * a) * ph * Wp
        # what enters each cell across its two d-faces
        fl = [ap - F, _roll(am + F, -1, d)]
        out = out - lam[d] * ik * (fl[0] + fl[1])
        del W, s, am, ap, F
        if nd == 2:
            e = 1 - d
            cx = [ctx, _roll(ctx, -1, d) if ctx is not None else None]
            bm, bp = torch.zeros_like(Q), torch.zeros_like(Q)
            for f, c in zip(fl, cx):
                m_, p_ = S.trans(d, c, f, A)
                bm, bp = bm + m_ * ik, bp + p_ * ik
            G = -0.5 * lam[d] * (bm + _roll(bp, 1, e))  # lower e-face of each cell
            out = out - lam[e] * ik * (_roll(G, -1, e) - G)
        elif nd == 3:
            f = fl[0] + fl[1]
            for g in range(3):
                if g == d:
                    continue
                e = 3 - d - g
                em, ep = S.split(e, f)
                a = (-0.5 * lam[d] * f + lam[d] * lam[e] / 6.0 *
                     (ep - em - _roll(ep, 1, e) + _roll(em, -1, e)))
                gm, gp = S.split(g, a)
                G = gm + _roll(gp, 1, g)
                out = out - lam[g] * (_roll(G, -1, g) - G)
    return _inner(out, nd, 2).contiguous(), speeds


def _weno5(v, eps=1e-6):
    """Left-biased value at the right edge of the third of five cell averages."""
    a, b, c, d, e = v
    b0 = 13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
    b1 = 13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
    b2 = 13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
    w0, w1, w2 = 0.1 / (eps + b0) ** 2, 0.6 / (eps + b1) ** 2, 0.3 / (eps + b2) ** 2
    return (w0 * (2 * a - 7 * b + 11 * c) + w1 * (2 * d + 5 * c - b) +
            w2 * (2 * c + 5 * d - e)) / (6 * (w0 + w1 + w2))


def _sharp_L(S, spec, q):
    """(L(Q), per-direction largest speeds) of the SharpClaw semi-discretisation."""
    Q, dx, L, speeds = _ghosts(q, 3, spec), _dx(spec), torch.zeros_like(q), []
    for d in range(2):
        n, t, e = 1 + d, 2 - d, 1 - d
        ax, N = 2 - d, spec["n"][d]
        X = Q.narrow(2 - e, 3, spec["n"][e])
        cell = [X.narrow(ax, k, N + 1) for k in range(6)]
        un, ut, H, c = S.roe(d, cell[2], cell[3])
        w = [S.coef(un, ut, H, c, v[0], v[n], v[t], v[3]) for v in cell]
        um = [_weno5([w[k][p] for k in (0, 1, 2, 3, 4)]) for p in range(4)]
        up = [_weno5([w[k][p] for k in (5, 4, 3, 2, 1)]) for p in range(4)]
        qm = S.assemble(un, ut, H, c, um, n, t, cell[0])  # right edge of the cell below
        qp = S.assemble(un, ut, H, c, up, n, t, cell[0])  # left edge of the cell above
        _, s, am, ap, _ = S.solve(d, qm, qp, None, None)
        speeds.append(max(float(si.abs().max()) for si in s))
        adq = S.flux(d, qm.narrow(ax, 1, N)) - S.flux(d, qp.narrow(ax, 0, N))
        L = L - (ap.narrow(ax, 0, N) + am.narrow(ax, 1, N) + adq) / dx[d]
    return L, speeds


def _sharp_step(S, spec, q, dt):
    L, s0 = _sharp_L(S, spec, q)
    q1 = q + dt * L
    L, s1 = _sharp_L(S, spec, q1)
    q2 = 0.75 * q + 0.25 * (q1 + dt * L)
    L, s2 = _sharp_L(S, spec, q2)
    return q / 3.0 + 2.0 / 3.0 * (q2 + dt * L), [max(v) for v in zip(s0, s1, s2)]


def _source(S, spec, q, dt):
    """The axisymmetric source over dt by Heun's method."""
    ny = spec["n"][1]
    r = _centers(spec["lower"][1], spec["upper"][1], ny)[:, None]

    def psi(q):
        f, v = torch.zeros_like(q), q[2] / q[0]
        f[0], f[1], f[2] = -q[2] / r, -q[1] * v / r, -q[2] * v / r
        f[3] = -(q[3] + S.pressure(q)) * v / r
        return f

    q1 = q + dt * psi(q)
    return 0.5 * (q + q1 + dt * psi(q1))


def _evolve(spec, q, aux, t_end, max_steps):
    """Steps with CFL control; (state, steps, rejects)."""
    S, dx = _system(spec), _dx(spec)
    sharp, src = spec["scheme"] == "sharpclaw", spec.get("source", "none") != "none"
    strang = spec.get("source_split", "godunov") == "strang"
    # first dt: speeds of first-order solves on the cell averages
    Q = _ghosts(q, 2, spec)
    A = _ghosts(aux, 2, spec, aux=True) if aux is not None else None
    kap = A[spec["capa_index"]] if spec.get("capa_index", -1) >= 0 else None
    rate = 0.0
    for d in range(spec["ndim"]):
        _, s, _, _, _ = S.solve(d, _roll(Q, 1, d), Q, _roll(A, 1, d) if A is not None else None, A)
        rate = max(rate, _face_speed(s, kap, d, spec["ndim"]) / dx[d])
    del Q
    dt, t, steps, rejects = spec["cfl_desired"] / rate, 0.0, 0, 0
    while t < t_end and steps < max_steps:
        final = t + dt >= t_end
        if final:
            dt = t_end - t
        q0 = _source(S, spec, q, 0.5 * dt) if src and strang else q
        new, speeds = (_sharp_step(S, spec, q0, dt) if sharp
                       else _classic_step(S, spec, q0, aux, dt))
        nu = max(dt * s / h for s, h in zip(speeds, dx))
        used, dt = dt, dt * spec["cfl_desired"] / nu
        if nu > spec["cfl_max"]:
            rejects += 1
            continue
        q = _source(S, spec, new, 0.5 * used if strang else used) if src else new
        t = t_end if final else t + used
        steps += 1
    return q, steps, rejects


def exact(case, seed):
    f64 = torch.float64
    if case["kind"] == "ensemble":
        specs, flat = _ensemble_inputs(case, seed)
        out, at = torch.zeros_like(flat, dtype=f64), 0
        for s in specs:
            q, _, _ = _evolve(s, s["q0"].to(f64), s["aux"].to(f64), FAR, case["steps"])
            n = q.numel()
            out[at:at + n] = q.reshape(-1)
            at += -(-n // 128) * 128
        return out
    if case["kind"] == "serve":
        return [_evolve(s, torch.from_numpy(s["q0"]).cuda().to(f64), None, s["t_end"], 10 ** 6)[0]
                for s in _serve_inputs(case, seed)]
    spec, q0, aux = _grid_inputs(case, seed)
    q, _, _ = _evolve(spec, q0.to(f64), aux.to(f64) if aux is not None else None, FAR,
                      case["steps"])
    return {"q": q, "steps": None, "rejects": None}
