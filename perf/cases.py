"""The work that a user of this library has it do, as timed cases.

Every case goes through the public entry points: joint solves (one call from zero models to the
result), the sensitivity products A m and A^T r of both fields, their autograd form, the Gramian,
and a batch of uneven inversions.  ``exact`` restates the same mathematics in plain torch, in 64
bits: closed-form prism fields near the stations, Gauss-Legendre cubature beyond eight cell sizes,
one library FFT per layer, and the reweighted conjugate gradient loop step by step.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2112_15562_gb300 as gj

FAR = 8.0  # prisms farther than this many of their largest sides are integrated by cubature
GRAV_UNIT = 6.6743e-11 * 1.0e3 * 1.0e5  # mGal per g/cc
FIELD = (50000.0, 60.0, 10.0)  # inducing field: nT, inclination, declination (degrees)


# ---------------------------------------------------------------------------------------------
# cases

def _case(kind, nx, ny, nz, precision="fp32", npad=(0, 0), sx=0, sy=0, off=(0, 0), cell=100.0, **more):
    c = dict(kind=kind, precision=precision, nx=nx, ny=ny, nz=nz, sx=sx or nx, sy=sy or ny, off_x=off[0], off_y=off[1],
             cell=cell, npad_y=npad[0], npad_x=npad[1])
    c.update(more)
    return c


def listed():
    named = lambda name, c: dict(c, name=name)  # noqa: E731
    return [
        # the paper-style toy inversion in full double precision, 50 iterations: the smallest
        # problem anybody solves, where launches and latency are everything
        named("solve-16x16x8-fp64", _case("solve", 16, 16, 8, "fp64", cell=50.0, iters=50, p=1, lam1=50.0, lam2=1500.0)),
        # a small survey of the paper's shape (50 x 30 stations, 10 layers), default padding
        named("solve-50x30x10-fp32", _case("solve", 50, 30, 10, iters=20, p=1, lam1=2.0, lam2=100.0)),
        # the paper's real-data shape (146 x 148 stations, 20 layers), default padding (294 x 300 points)
        named("solve-146x148x20-fp32", _case("solve", 148, 146, 20, iters=20, p=1, lam1=2.0, lam2=100.0)),
        # the headline workload: a joint inversion of 256 x 256 stations and 2.6 million cells a model
        named("solve-256x256x40-fp32", _case("solve", 256, 256, 40, iters=20, p=1, lam1=2.0, lam2=100.0)),
        # predicted data of both fields from the headline workload's models
        named("forward-256x256x40-fp32", _case("forward", 256, 256, 40)),
        # gradients of both fields on an odd, ragged grid with padding prisms around the stations
        named("adjoint-251x243x37-fp32", _case("adjoint", 251, 243, 37, npad=(512, 512), sx=213, sy=201, off=(19, 21))),
        # the operator benchmark's grid at its circulant size 255 (= 3 5 17), as the library pads it
        named("products-128x128x32-fp32", _case("both", 128, 128, 32, cell=50.0)),
        # forward and adjoint of the headline grid in double precision, the reference form
        named("products-256x256x40-fp64", _case("both", 256, 256, 40, "fp64")),
        # a learning or sensitivity loop on a large grid: forward and backward of both fields
        named("autograd-512x512x48-fp32", _case("autograd", 512, 512, 48)),
        # the same where the spectra do not fit beside the rest: each layer's is rebuilt in every product
        named("recompute-512x512x48-fp32", _case("recompute", 512, 512, 48)),
        # six uneven surveys inverted together by one graph
        named("batch-6-uneven-fp32", _case("batch", 256, 256, 40, iters=10, p=1, lam1=2.0, lam2=100.0, count=6, sizes=4)),
        # the coupling term and its directions for the headline workload's models
        named("gramian-2.6M-fp32", _case("gramian", 256, 256, 40)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "forward", "adjoint", "both", "both", "autograd", "gramian", "recompute", "batch"])
    precision = "fp64" if kind in ("solve", "forward", "adjoint", "both", "gramian") and rng.random() < 0.3 else "fp32"
    if kind == "batch":
        return _case("batch", 192, 192, 24, iters=rng.randint(4, 10), p=1, lam1=2.0, lam2=100.0, count=rng.randint(2, 5),
                     sizes=rng.randint(10, 10 ** 6))
    top = 256 if precision == "fp32" else 160
    if kind == "autograd":
        nx, ny, nz = rng.randint(120, 512), rng.randint(120, 512), rng.randint(4, 32)
    elif kind == "recompute":
        nx, ny, nz = _log_int(rng, 24, 300), _log_int(rng, 24, 300), rng.randint(3, 12)
    else:
        nx, ny, nz = _log_int(rng, 12, top), _log_int(rng, 12, top), rng.randint(3, 40)
    sx, sy, off = nx, ny, (0, 0)
    if kind in ("forward", "adjoint", "both", "autograd") and rng.random() < 0.4:  # padding prisms
        ox, oy = rng.randint(0, nx // 6), rng.randint(0, ny // 6)
        sx, sy, off = nx - 2 * ox - rng.randint(0, 1), ny - 2 * oy - rng.randint(0, 1), (ox, oy)
    npad = (0, 0)
    if precision == "fp32" and kind != "recompute" and rng.random() < 0.6:  # the sizes of the warp transforms
        if max(nx, ny) <= 256:
            npad = (256, 512) if ny <= 128 and rng.random() < 0.7 else (512, 512)
        elif kind == "autograd":
            npad = (1024, 1024)
    more = {}
    if kind == "solve":
        more = dict(iters=rng.randint(4, 20), p=rng.choice([1, 1, 2]), lam1=2.0, lam2=100.0)
    return _case(kind, nx, ny, nz, precision, npad, sx, sy, off, rng.choice([50.0, 100.0]), **more)


# ---------------------------------------------------------------------------------------------
# inputs

class _Grid:
    def __init__(self, c, nx=None, ny=None, nz=None):
        self.nx, self.ny, self.nz = nx or c["nx"], ny or c["ny"], nz or c["nz"]
        self.sx, self.sy = (c["sx"], c["sy"]) if nx is None else (nx, ny)
        self.off_x, self.off_y = (c["off_x"], c["off_y"]) if nx is None else (0, 0)
        self.dx = self.dy = float(c["cell"])
        self.z_edges = np.arange(self.nz + 1, dtype=np.float64) * self.dx
        self.station_z = 0.0
        self.n, self.s = self.nx * self.ny * self.nz, self.sx * self.sy


class _Mag:
    F, incl, decl = FIELD


def _dtype(c):
    return torch.float64 if c["precision"] == "fp64" else torch.float32


def _rand(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _model(g, vmax, seed, dtype):
    """A smooth field and six boxes, in [0, vmax]."""
    gen = _rand(seed)
    coarse = torch.rand((1, 1, max(2, g.nz // 6), max(2, g.ny // 12), max(2, g.nx // 12)), generator=gen, device="cuda", dtype=torch.float64)
    m = 0.6 * torch.nn.functional.interpolate(coarse, size=(g.nz, g.ny, g.nx), mode="trilinear", align_corners=True)[0, 0]
    rs = np.random.RandomState(seed % (1 << 31))
    for _ in range(6):
        w = [max(1, int(v * rs.uniform(0.06, 0.25))) for v in (g.nx, g.ny, g.nz)]
        at = [rs.randint(0, v - k + 1) for v, k in zip((g.nx, g.ny, g.nz), w)]
        m[at[2]:at[2] + w[2], at[1]:at[1] + w[1], at[0]:at[0] + w[0]] += 0.4
    return (m.clamp_(0.0, 1.0) * vmax).reshape(-1).to(dtype).contiguous()


def _boxes(g, seed):
    """Three dipping bodies, sheared one cell per layer, as boxes (x0, x1, y0, y1, z0, z1) in metres."""
    rs = np.random.RandomState(seed % (1 << 31))
    lo = max(2, min(g.nx, g.ny) // 12)
    hi = max(lo + 1, min(g.nx, g.ny) // 4)
    out = []
    for _ in range(3):
        wx, wy = rs.randint(lo, hi + 1), rs.randint(lo, hi + 1)
        top, thick = rs.randint(1, max(2, g.nz // 4)), rs.randint(max(2, g.nz // 8), max(3, g.nz // 2))
        x0, y0 = rs.randint(0, max(1, g.nx - wx - thick)), rs.randint(0, max(1, g.ny - wy))
        for r in range(top, min(g.nz, top + thick)):
            xa, xb = x0 + r - top, min(g.nx, x0 + r - top + wx)
            if xb > xa:
                out.append((xa * g.dx, xb * g.dx, y0 * g.dy, (y0 + wy) * g.dy, g.z_edges[r], g.z_edges[r + 1]))
    return out


def _survey(g, seed, dtype):
    """Observed data and their standard deviations: the closed-form fields of the bodies, with one per cent noise and a floor."""
    jx = (torch.arange(g.sx, device="cuda", dtype=torch.float64) + g.off_x + 0.5) * g.dx
    jy = (torch.arange(g.sy, device="cuda", dtype=torch.float64) + g.off_y + 0.5) * g.dy
    bodies = _boxes(g, seed)
    dobs, sigma = [], []
    gen = _rand(seed + 7)
    for field, value in ((0, 1.0), (1, 0.1)):
        d = torch.zeros((g.sy, g.sx), device="cuda", dtype=torch.float64)
        for x0, x1, y0, y1, z0, z1 in bodies:
            u = [(x - jx)[None, :].expand(g.sy, g.sx) for x in (x0, x1)]
            v = [(y - jy)[:, None].expand(g.sy, g.sx) for y in (y0, y1)]
            d += value * _closed(field, u, v, [torch.full_like(d, z - g.station_z) for z in (z0, z1)])
        sg = 0.01 * d.abs() + 0.01 * d.abs().max()
        d = d + sg * torch.randn(d.shape, generator=gen, device="cuda", dtype=torch.float64)
        dobs.append(d.reshape(-1).to(dtype).contiguous())
        sigma.append(sg.reshape(-1).to(dtype).contiguous())
    return dobs, sigma


def _depth(g, dtype):
    z = 0.5 * (g.z_edges[:-1] + g.z_edges[1:])
    return [torch.from_numpy((z / z[0]) ** (-b / 2.0)).to(device="cuda", dtype=dtype) for b in (2.0, 3.0)]


def _batch_grids(c):
    rs = np.random.RandomState(c["sizes"] % (1 << 31))
    out = []
    for _ in range(c["count"]):
        nx, ny = (int(rs.randint(4, c["nx"] // 16 + 1)) * 16 for _ in range(2))
        out.append(_Grid(c, nx, ny, int(rs.randint(min(16, c["nz"]), c["nz"] + 1))))
    return out


def _inputs(c, seed):
    dt = _dtype(c)
    if c["kind"] == "batch":
        return [(g, *_survey(g, seed + 31 * i, dt), _depth(g, dt)) for i, g in enumerate(_batch_grids(c))]
    g = _Grid(c)
    if c["kind"] == "solve":
        return (g, *_survey(g, seed, dt), _depth(g, dt))
    m = [_model(g, 1.0, seed, dt), _model(g, 0.1, seed + 1000, dt)]
    if c["kind"] == "gramian":
        return g, m, None
    gen = _rand(seed + 5)
    r = [torch.randn(g.s, generator=gen, device="cuda", dtype=torch.float64).to(dt) for _ in range(2)]
    return g, m, r


def _params(c):
    return gj.solver_params(p=(c["p"], c["p"]), alpha1=(2e4, 2e4), q=(0.95, 0.95), alpha_min=(5.0, 20.0), lam=(c["lam1"], c["lam2"]),
                            lo=(0.0, 0.0), hi=(1.0, 0.1), kmax=c["iters"], stop_on_chi2=False)


def _ops(c, g, npad, recompute=False):
    return [gj.bttb_setup(g, "gravity", precision=c["precision"], npad=npad, recompute=recompute),
            gj.bttb_setup(g, "magnetic", _Mag, precision=c["precision"], npad=npad, recompute=recompute)]


def prepare(case, seed):
    c = case
    given = _inputs(c, seed)
    if c["kind"] == "batch":
        ops = [_ops(c, g, (256 if g.ny <= 128 else 512, 512)) for g, *_ in given]
    elif c["kind"] == "gramian":
        ops = None
    else:
        ops = _ops(c, given[0], (c["npad_y"], c["npad_x"]), c["kind"] == "recompute")
    return {"case": c, "given": given, "ops": ops}


# ---------------------------------------------------------------------------------------------
# one pass

def run(state):
    c, given, ops = state["case"], state["given"], state["ops"]
    kind = c["kind"]
    if kind == "solve":
        g, dobs, sigma, depth = given
        m = [torch.zeros(g.n, dtype=o.dtype, device="cuda") for o in ops]
        rep = gj.rrcg_joint_solve(ops, _params(c), dobs, sigma, depth, m)
        return {"m": m, "phi": rep["phi"], "alpha": rep["alpha"], "iterations": rep["iterations"]}
    if kind == "batch":
        models, solvers = [], []
        for (g, dobs, sigma, depth), o in zip(given, ops):
            m = [torch.zeros(g.n, dtype=o[0].dtype, device="cuda") for _ in range(2)]
            models.append(m)
            solvers.append(gj.Solver(o, _params(c), dobs, sigma, depth, m))
        together = gj.Batch(solvers)
        together.step(c["iters"])
        together.close()
        for s in solvers:
            s.close()
        return {"m": models}
    g, m, r = given
    if kind == "gramian":
        S, l1, l2 = gj.gramian_value_grad(m[0], m[1])
        return {"S": S.to(m[0].dtype), "l": [l1, l2]}  # the term joins an objective in the models' precision
    if kind in ("autograd", "recompute"):
        d, grad = [], []
        for i in range(2):
            x = m[i].detach().requires_grad_(True)
            y = gj.G(ops[i], x)
            y.backward(r[i])
            d.append(y.detach())
            grad.append(x.grad)
        return {"d": d, "g": grad}
    out = {}
    if kind in ("forward", "both"):
        out["d"] = gj.g_forward_pair(ops, m)
    if kind in ("adjoint", "both"):
        out["g"] = gj.g_adjoint_pair(ops, r)
    return out


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without

def _smooth(n):
    while True:
        k = n
        for p in (2, 3, 5, 7):
            while k % p == 0:
                k //= p
        if k == 1:
            return n
        n += 1


def _product_work(g, es, npad_y=0, npad_x=0, stored=True):
    """One product of both fields: vectors in and out, the spectra once (the gravity one real where the
    stations cover the prisms), real 2-D transforms of every layer and one of the data."""
    Ny, Nx = npad_y or _smooth(g.sy + g.ny - 1), npad_x or _smooth(g.sx + g.nx - 1)
    ncol = Nx // 2 + 1
    even = (g.sx, g.sy, g.off_x, g.off_y) == (g.nx, g.ny, 0, 0)
    spec = (g.nz * ncol * (Ny * 2 + ((Ny // 2 + 1) if even else 2 * Ny)) * es) if stored else 0
    fft = 2.5 * Nx * Ny * math.log2(Nx * Ny)
    return 2 * (g.n + g.s) * es + spec, 2 * ((g.nz + 1) * fft + g.nz * 8.0 * ncol * Ny)


def _solve_work(g, c, es, npad_y=0, npad_x=0):
    b, f = _product_work(g, es, npad_y, npad_x)
    b -= 2 * (g.n + g.s) * es
    # an iteration: m, p -> m; m -> l; l, p, m -> p, and the data vectors
    it_b = 3 * b + 2 * es * (9 * g.n + 4 * g.s)
    return c["iters"] * it_b + b, c["iters"] * (3 * f + 60.0 * g.n) + f


def work(case):
    c = case
    es = 8 if c["precision"] == "fp64" else 4
    if c["kind"] == "batch":
        parts = [_solve_work(g, c, es, 256 if g.ny <= 128 else 512, 512) for g in _batch_grids(c)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    g = _Grid(c)
    if c["kind"] == "solve":
        b, f = _solve_work(g, c, es, c["npad_y"], c["npad_x"])
        return {"bytes": b, "flops": f}
    if c["kind"] == "gramian":
        return {"bytes": 4 * g.n * es, "flops": 18 * g.n}
    b, f = _product_work(g, es, c["npad_y"], c["npad_x"], c["kind"] != "recompute")
    k = 2 if c["kind"] in ("both", "autograd", "recompute") else 1
    if c["kind"] == "recompute":  # the tables (27 cubature points an entry, mostly) and their transforms
        entries = (g.sx + g.nx - 1) * (g.sy + g.ny - 1) * g.nz
        f += 2 * entries * 27 * 20.0 + f
    return {"bytes": k * b, "flops": k * f}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits

def _direction():
    i, d = math.radians(FIELD[1]), math.radians(FIELD[2])
    return math.cos(i) * math.sin(d), math.cos(i) * math.cos(d), math.sin(i)


def _log_sum(a, R, bc):
    """log(a + R), R = sqrt(a^2 + bc), without the cancellation at negative a."""
    return torch.where(a >= 0, torch.log(torch.where(a >= 0, a + R, 1.0)), torch.log(torch.where(a < 0, bc / torch.where(a < 0, R - a, 1.0), 1.0)))


def _closed(field, u, v, w):
    """The prism's field at its eight corners (lower, upper) relative to the station: u East, v North, w down."""
    t = _direction()
    total = 0.0
    for i in range(2):
        for j in range(2):
            for k in range(2):
                x, y, z = u[i], v[j], w[k]
                R = torch.sqrt(x * x + y * y + z * z)
                if field == 0:
                    f = z * torch.atan2(x * y, z * R) - x * _log_sum(y, R, x * x + z * z) - y * _log_sum(x, R, y * y + z * z)
                else:
                    f = -(t[0] ** 2 * torch.atan(y * z / (x * R)) + t[1] ** 2 * torch.atan(x * z / (y * R)) + t[2] ** 2 * torch.atan2(x * y, z * R))
                    f = f + 2 * (t[0] * t[1] * _log_sum(z, R, x * x + y * y) + t[0] * t[2] * _log_sum(y, R, x * x + z * z)
                                 + t[1] * t[2] * _log_sum(x, R, y * y + z * z))
                total = total + (f if (i + j + k) % 2 else -f)  # (-1)^(i + j + k) with the limits numbered 1 and 2
    return total * (GRAV_UNIT if field == 0 else FIELD[0] / (4 * math.pi))


def _cubature(field, uc, vc, wc, h, hw):
    t = _direction()
    x, wt = np.polynomial.legendre.leggauss(5)
    total = torch.zeros_like(uc)
    for i in range(5):
        u = uc + h * x[i]
        for j in range(5):
            v = vc + h * x[j]
            for k in range(5):
                w = wc + hw * x[k]
                r2 = u * u + v * v + w * w
                if field == 0:
                    f = w / (r2 * torch.sqrt(r2))
                else:
                    tr = t[0] * u + t[1] * v + t[2] * w
                    f = (3 * tr * tr - r2) / (r2 * r2 * torch.sqrt(r2))
                total += wt[i] * wt[j] * wt[k] * f
    return total * (h * h * hw) * (GRAV_UNIT if field == 0 else FIELD[0] / (4 * math.pi))


class _Exact:
    """One field's operator in 64 bits: the layers' spectra of the circulant embedding."""

    def __init__(self, g, field):
        self.g = g
        self.shape = _smooth(g.sy + g.ny - 1), _smooth(g.sx + g.nx - 1)
        f64 = dict(device="cuda", dtype=torch.float64)
        cy = torch.arange(-(g.ny - 1), g.sy, device="cuda")
        cx = torch.arange(-(g.nx - 1), g.sx, device="cuda")
        vc = (-(cy + g.off_y).to(torch.float64) * g.dy)[:, None].expand(len(cy), len(cx)).contiguous()
        uc = (-(cx + g.off_x).to(torch.float64) * g.dx)[None, :].expand(len(cy), len(cx)).contiguous()
        self.spec = []
        h = 0.5 * g.dx
        for r in range(g.nz):
            z0, z1 = float(g.z_edges[r]) - g.station_z, float(g.z_edges[r + 1]) - g.station_z
            wc, hw = 0.5 * (z0 + z1), 0.5 * (z1 - z0)
            K = _cubature(field, uc, vc, torch.full_like(uc, wc), h, hw)
            near = uc * uc + vc * vc + wc * wc < (FAR * max(g.dx, z1 - z0)) ** 2
            if bool(near.any()):
                u, v = uc[near], vc[near]
                K[near] = _closed(field, [u - h, u + h], [v - h, v + h], [torch.full_like(u, z0), torch.full_like(u, z1)])
            T = torch.zeros(self.shape, **f64)
            T[(cy % self.shape[0])[:, None], (cx % self.shape[1])[None, :]] = K
            self.spec.append(torch.fft.rfft2(T))

    def forward(self, m):
        g = self.g
        m = m.reshape(g.nz, g.ny, g.nx)
        Y = 0.0
        for r in range(g.nz):
            Y = Y + self.spec[r] * torch.fft.rfft2(m[r], s=self.shape)
        return torch.fft.irfft2(Y, s=self.shape)[:g.sy, :g.sx].reshape(-1)

    def adjoint(self, d):
        g = self.g
        V = torch.fft.rfft2(d.reshape(g.sy, g.sx), s=self.shape)
        return torch.stack([torch.fft.irfft2(T.conj() * V, s=self.shape)[:g.ny, :g.nx].reshape(-1) for T in self.spec]).reshape(-1)


def _exact_solve(g, c, dobs, sigma, depth):
    A = [_Exact(g, 0), _Exact(g, 1)]
    dob, wd = [x.double() for x in dobs], [1.0 / x.double() for x in sigma]
    ws = [x.double().repeat_interleave(g.nx * g.ny) for x in depth]
    lam, lo, hi, q, least = (c["lam1"], c["lam2"]), (0.0, 0.0), (1.0, 0.1), 0.95, (5.0, 20.0)
    target = g.s + math.sqrt(2.0 * g.s)
    m = [torch.zeros(g.n, device="cuda", dtype=torch.float64) for _ in range(2)]
    alpha, sat, before, ll_before, k = [2e4, 2e4], [False, False], None, None, 0
    own = lam == (0.0, 0.0)
    while True:
        rt = [wd[i] * (A[i].forward(m[i]) - dob[i]) for i in range(2)]
        phi = [float(x @ x) for x in rt]
        for i in range(2):
            sat[i] = sat[i] or phi[i] <= target
            if k and not sat[i]:
                alpha[i] = max(q * alpha[i], least[i])
        if k == c["iters"]:
            return {"m": m, "phi": phi, "alpha": alpha, "iterations": None}
        W = [ws[i] * ((m[i] ** 2 + 1e-9) ** ((c["p"] - 2) / 4.0)) for i in range(2)]
        a, b, ab = float(m[0] @ m[0]), float(m[1] @ m[1]), float(m[0] @ m[1])
        lG = [b * m[0] - ab * m[1], a * m[1] - ab * m[0]]
        step = [A[i].adjoint(wd[i] * rt[i]) / W[i] + alpha[i] * W[i] * m[i] + lam[i] * lG[i] for i in range(2)]
        ll = [float(x @ x) for x in step]
        if before is None:
            p = step
        elif own:
            p = [step[i] + ll[i] / ll_before[i] * before[i] for i in range(2)]
        else:
            p = [step[i] + sum(ll) / sum(ll_before) * before[i] for i in range(2)]
        x = [wd[i] * A[i].forward(p[i] / W[i]) for i in range(2)]
        num = [float(p[i] @ step[i]) for i in range(2)]
        den = [float(x[i] @ x[i]) + (alpha[i] + lam[i]) * float(p[i] @ p[i]) for i in range(2)]
        s = [num[i] / den[i] for i in range(2)] if own else [sum(num) / sum(den)] * 2
        m = [torch.clamp(m[i] - s[i] * p[i] / W[i], lo[i], hi[i]) for i in range(2)]
        before, ll_before, k = p, ll, k + 1


def exact(case, seed):
    c = case
    given = _inputs(c, seed)
    if c["kind"] == "batch":
        return {"m": [_exact_solve(g, c, dobs, sigma, depth)["m"] for g, dobs, sigma, depth in given]}
    if c["kind"] == "solve":
        return _exact_solve(given[0], c, *given[1:])
    g, m, r = given
    m = [x.double() for x in m]
    if c["kind"] == "gramian":
        a, b, ab = m[0] @ m[0], m[1] @ m[1], m[0] @ m[1]
        rest = m[1] - ab / a * m[0]
        return {"S": (a * (rest @ rest)).reshape(1), "l": [b * m[0] - ab * m[1], a * m[1] - ab * m[0]]}
    out = {"d": [], "g": []}
    for i in range(2):
        A = _Exact(g, i)
        if c["kind"] != "adjoint":
            out["d"].append(A.forward(m[i]))
        if c["kind"] != "forward":
            out["g"].append(A.adjoint(r[i].double()))
    return {k: v for k, v in out.items() if v}
