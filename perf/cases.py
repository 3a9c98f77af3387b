"""The work that is timed: runs of the solver through its Python entry points.

A case is one program's pass.  ``prepare`` builds what such a program holds
(the solver with its bed and boundaries, the initial state on the GPU), and
``run`` sets the state, steps, and reads back what the program wants: the
fields, the gauge records, the run-up field, an ensemble's fields, a gauge
misfit's gradients, or rendered frames.  Every pass starts from the same given
state, so its outputs depend on the case and the seed alone (the makers' time
runs on from pass to pass).

Sizes and settings are those of the workloads in
``paper_1611_05984_gb300/scenarios.py`` and of the benchmark: the solitary-wave
channel, the beach with shoals at 2048 x 2048 in both precisions and at
8192 x 8192 under directional waves, the ensemble of uneven beaches, the
512 x 512 gauge-misfit gradient, and the paper's tank geometries (planar beach,
semicircular shoal, conical island).  The inputs are seeded here: shoals,
crests and wave trains of random place, height, period and direction, so that
the whole water carries waves and the shoreline moves, as in a run under way.

``exact`` computes the same passes in plain torch in 64 bits, from the
equations alone (KP07 reconstruction and central-upwind fluxes, Eq. 9-13 and
31-32 of arXiv 1611.05984 on the right side, Eq. 15-23 in time, boundaries of
Eq. 24-30), with the line systems solved by cyclic reduction; the gradients
come from autograd.
"""
import math
import random

import torch
from torch.utils.checkpoint import checkpoint

from paper_1611_05984_gb300 import celeris

G = 9.81
BD = 1.0 / 15.0
THETA = 1.3
W, E, S, N = celeris.WEST, celeris.EAST, celeris.SOUTH, celeris.NORTH


# ------------------------------------------------------------------ the cases

def _case(name, task, bed, nx, ny, dx, steps, dtype="f32", K=1, model="bsnq", friction="manning", **more):
    c = dict(name=name, task=task, bed=bed, nx=nx, ny=ny, dx=dx, steps=steps, dtype=dtype, K=K, model=model,
             friction=friction)
    c.update(more)
    return c


def listed():
    return [
        # the smallest run: a solitary wave in a walled channel, predictor only, double precision (validation runs)
        _case("channel_f64", "fields", "channel", 256, 32, 0.05, 24, "f64", K=0, friction="none"),
        # solitary-wave run-up on a planar beach, one depth wide: a few thousand cells, latency alone
        _case("planar_beach", "runup", "planar", 559, 4, 0.25, 24, friction="quadratic"),
        # regular waves over a semicircular shoal, gauges along the tank recorded every step
        _case("shoal_gauges", "gauges", "shoal", 2000, 65, 0.0175, 24, friction="none"),
        # a solitary wave on a conical island, run-up tracked; odd sizes, no friction
        _case("island_runup", "runup", "island", 601, 601, 0.05, 16, friction="none"),
        # a shallow-water run (no dispersive solves) of a ragged beach, quadratic friction
        _case("beach_nlsw", "fields", "beach", 1000, 750, 1.0, 16, model="nlsw", friction="quadratic"),
        # the main workload, single and double precision
        _case("beach_2048_f32", "fields", "beach", 2048, 2048, 1.0, 16),
        _case("beach_2048_f64", "fields", "beach", 2048, 2048, 1.0, 4, "f64"),
        # the largest grid, three wave trains of random direction
        _case("beach_8192_f32", "fields", "directional", 8192, 8192, 1.0, 6),
        # many uneven scenarios stepped together
        _case("ensemble_40", "ensemble", "beach", 1024, 512, 1.0, 14, members=40),
        # gradient of a gauge misfit with respect to the surface and the bed, recomputed from checkpoints
        _case("gradient_512_f32", "gradient", "hump", 512, 512, 1.0, 60, every=20),
        # the same in double precision on a ragged grid, every step kept
        _case("gradient_f64", "gradient", "hump", 200, 150, 1.0, 24, "f64", every=0),
        # frames of a stored snapshot: water shaded by the Fresnel equations, the surface, the speed
        _case("frames_2048", "frames", "beach", 2048, 2048, 1.0, 3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    task = rng.choice(["fields", "fields", "fields", "fields", "gauges", "runup", "ensemble", "gradient", "frames"])
    dtype = rng.choice(["f32", "f32", "f32", "f64"])
    friction = rng.choice(["manning", "manning", "quadratic", "none"])
    if task == "ensemble":
        nx, ny = _log_int(rng, 128, 1024), _log_int(rng, 128, 512)
        return dict(task=task, bed="beach", nx=nx, ny=ny, dx=1.0, steps=rng.randint(10, 20), dtype=dtype,
                    K=1, model="bsnq", friction=friction, members=rng.randint(3, 40 if dtype == "f32" else 6))
    if task == "gradient":
        nx, ny = _log_int(rng, 64, 512 if dtype == "f32" else 200), _log_int(rng, 64, 512 if dtype == "f32" else 200)
        steps = rng.randint(12, 40)
        return dict(task=task, bed="hump", nx=nx, ny=ny, dx=1.0, steps=steps, dtype=dtype, K=1,
                    model=rng.choice(["bsnq", "bsnq", "bsnq", "nlsw"]), friction=friction,
                    every=rng.choice([0, rng.randint(5, steps)]))
    if task in ("gauges", "runup"):
        bed = rng.choice(["shoal", "beach"]) if task == "gauges" else rng.choice(["island", "planar"])
        if bed == "planar":
            nx, ny, dx = _log_int(rng, 450, 1600), rng.randint(4, 40), 0.25
        elif bed == "shoal":
            ny = rng.randint(33, 130)
            nx = _log_int(rng, 1000, 4000)
            dx = 35.0 / nx
        elif bed == "island":
            nx = ny = _log_int(rng, 201, 1201)
            dx = 30.0 / nx
        else:
            nx, ny, dx = _log_int(rng, 100, 1500), _log_int(rng, 100, 1500), 1.0
        return dict(task=task, bed=bed, nx=nx, ny=ny, dx=dx, steps=rng.randint(6, 20), dtype=dtype, K=1,
                    model="bsnq", friction=friction if bed in ("planar", "beach") else "none")
    if task == "frames":
        nx, ny = _log_int(rng, 200, 3000), _log_int(rng, 200, 3000)
        return dict(task=task, bed="beach", nx=nx, ny=ny, dx=1.0, steps=rng.randint(1, 4), dtype=dtype, K=1,
                    model="bsnq", friction="manning")
    hi = 5000 if dtype == "f32" else 1500
    nx, ny = _log_int(rng, 64, hi), _log_int(rng, 32, hi)
    bed = rng.choice(["beach", "beach", "directional", "channel"])
    if bed == "channel":
        return dict(task=task, bed=bed, nx=max(nx, 200), ny=min(ny, 400), dx=0.05, steps=rng.randint(6, 24), dtype=dtype,
                    K=rng.choice([0, 2]), model="bsnq", friction="none")
    return dict(task=task, bed=bed, nx=nx, ny=ny, dx=1.0, steps=rng.randint(4, 16) if nx * ny < 4e6 else 4,
                dtype=dtype, K=1 if rng.random() < 0.8 else 3, model=rng.choice(["bsnq", "bsnq", "bsnq", "nlsw"]),
                friction=friction)


# ------------------------------------------------------------- seeded scenes

class Scene:
    """One scenario: bed, boundaries, parameters and initial state (64-bit
    device tensors rounded to the case's type)."""


def _soliton(x, H, d, x0, ramp=1.0):
    k = math.sqrt(3.0 * H / (4.0 * d ** 3))
    eta = H / torch.cosh(torch.clamp(k * (x - x0), -80.0, 80.0)) ** 2
    return eta, math.sqrt(G * (H + d)) * eta


def _scene(case, seed, nx=None, ny=None):
    rng = random.Random(int(seed) * 7919 + 17)
    nx, ny = nx or case["nx"], ny or case["ny"]
    s = Scene()
    s.nx, s.ny = nx, ny
    f = dict(dtype=torch.float64, device="cuda")
    bed = case["bed"]
    s.dx = s.dy = case["dx"]
    s.K, s.model = case["K"], {"bsnq": celeris.BSNQ, "nlsw": celeris.NLSW}[case["model"]]
    s.eps, s.ws = 1e-8, 0.0
    s.sides = {k: (celeris.SOLID, 0, ()) for k in (W, E, S, N)}
    s.friction, s.fcoef = {"none": (celeris.FRIC_NONE, 0.0), "quadratic": (celeris.FRIC_QUADRATIC, 0.005),
                           "manning": (celeris.FRIC_MANNING, 0.015)}[case["friction"]]
    s.delta = 1e-3
    Q = torch.zeros((ny, nx), **f)
    if bed in ("beach", "directional", "hump"):
        d0, cr = 10.0, 0.1
        # short grids get a coarser spacing, so that the beach's toe lies inside the grid
        s.dx = s.dy = max(case["dx"], math.ceil(d0 * 30.0 / (0.7 * nx) * 4.0) / 4.0)
        x = (torch.arange(nx, **f) + 0.5) * s.dx
        y = (torch.arange(ny, **f) + 0.5) * s.dy
        Lx, Ly = nx * s.dx, ny * s.dy
        z = torch.clamp((x - 0.85 * Lx) / 30.0, min=-d0).expand(ny, nx).clone()
        for _ in range(8):
            h, wd = rng.uniform(1.0, 4.0), rng.uniform(20.0, 80.0)
            cx, cy = rng.uniform(0.1, 0.75) * Lx, rng.uniform(0.1, 0.9) * Ly
            z += h * torch.outer(torch.exp(-((y - cy) / wd) ** 2), torch.exp(-((x - cx) / wd) ** 2))
        sponge = min(50, max(2, ny // 8))
        s.sides[S] = s.sides[N] = (celeris.SPONGE, sponge, ())
        if bed == "hump":
            s.sides[W] = (celeris.SPONGE, min(50, max(2, nx // 10)), ())
        else:
            n = 3 if bed == "directional" else 1
            s.sides[W] = (celeris.SINE, 0, tuple((0.3 / n, rng.uniform(6.0, 14.0), rng.uniform(-0.5, 0.5) if n > 1 else 0.0,
                                                  rng.uniform(0.0, 6.28)) for _ in range(n)))
        d = torch.clamp(-z, min=0.0)
        fade = torch.clamp(d / 4.0, max=1.0)
        eta = torch.zeros((ny, nx), **f)
        P = torch.zeros((ny, nx), **f)
        for _ in range(3):
            a, T, th, ph = rng.uniform(0.05, 0.15), rng.uniform(7.0, 14.0), rng.uniform(-0.6, 0.6), rng.uniform(0, 6.28)
            k0 = (2.0 * math.pi / T) ** 2 / G
            k = k0 / math.sqrt(math.tanh(k0 * d0))
            e = a * torch.sin(k * math.cos(th) * x[None, :] + k * math.sin(th) * y[:, None] + ph) * fade
            c = torch.sqrt(G * d)
            eta += e
            P += c * math.cos(th) * e
            Q += c * math.sin(th) * e
        if bed == "hump":
            r2 = ((x - rng.uniform(0.3, 0.5) * Lx) ** 2)[None, :] + ((y - rng.uniform(0.4, 0.6) * Ly) ** 2)[:, None]
            eta += 0.5 * torch.exp(-r2 / 30.0 ** 2) * fade
        w = eta
        depth = d0
    elif bed == "channel":
        cr, depth, s.eps = 0.2, 1.0, 5e-12
        z = torch.full((ny, nx), -1.0, **f)
        x = (torch.arange(nx, **f) + 0.5) * s.dx
        e, p = _soliton(x, rng.uniform(0.05, 0.12), 1.0, rng.uniform(0.3, 0.7) * nx * s.dx)
        w, P = e.expand(ny, nx).clone(), p.expand(ny, nx).clone()
    elif bed == "planar":
        cr, depth = 0.03 / case["dx"], 1.0
        H = rng.uniform(0.1, 0.3)
        L = nx * s.dx
        x = (torch.arange(nx, **f) + 0.5) * s.dx
        toe = L - 2.5 * 19.85
        z = torch.clamp(-1.0 + (x - toe) / 19.85, min=-1.0).expand(ny, nx).clone()
        e, p = _soliton(x, H, 1.0, toe + rng.uniform(0.0, 8.0))
        w, P = e.expand(ny, nx).clone(), p.expand(ny, nx).clone()
        s.sides[W] = (celeris.SPONGE, int(round(20.0 / s.dx)), ())
        s.delta = s.dx / 19.85 / 3.0
    elif bed == "shoal":
        s.dy = 6.096 / ny
        h0 = 0.4572
        x = (torch.arange(nx, **f) + 0.5) * s.dx
        y = (torch.arange(ny, **f) + 0.5) * s.dy
        gy = torch.sqrt(y * (6.096 - y))
        z = -h0 + torch.clamp((x[None, :] - 10.67 + gy[:, None]) / 25.0, 0.0, 0.3048)
        cr, depth = 0.12, h0
        a, T, ph = rng.uniform(0.005, 0.0075), rng.uniform(1.6, 2.6), rng.uniform(0.0, 6.28)
        k0 = (2.0 * math.pi / T) ** 2 / G
        k = k0 / math.sqrt(math.tanh(k0 * h0))
        w = (a * torch.sin(ph - k * x)).expand(ny, nx) + 0.001 * torch.outer(torch.cos(2.0 * y), torch.sin(1.3 * x + ph))
        P = (2.0 * math.pi / T / k) * w
        s.sides[W] = (celeris.SINE, 0, ((a, T, 0.0, ph),))
        s.sides[E] = (celeris.SPONGE, int(round(5.0 / s.dx)), ())
    else:   # the conical island
        d, cr = 0.32, 0.1
        x = (torch.arange(nx, **f) + 0.5) * s.dx
        y = (torch.arange(ny, **f) + 0.5) * s.dy
        r = torch.sqrt(((x - 15.0) ** 2)[None, :] + ((y - 15.0) ** 2)[:, None])
        z = -d + torch.clamp((3.6 - r) / 4.0, 0.0, 0.625)
        e, p = _soliton(x, rng.uniform(0.04, 0.18) * d, d, rng.uniform(11.0, 15.0))
        fade = torch.clamp(-z / d, 0.0, 1.0) ** 2
        w, P = e * fade, p * fade
        s.eps, depth = 1e-10, d
        s.sides[W] = s.sides[E] = (celeris.SPONGE, int(round(1.5 / s.dx)), ())
        s.delta = 0.25 * s.dx / 3.0
    s.dt = cr * min(s.dx, s.dy) / math.sqrt(G * depth)
    if bed == "shoal":
        s.dt = min(s.dt, 0.001)
    t = torch.float32 if case["dtype"] == "f32" else torch.float64
    s.dtype = t
    s.z, s.w, s.P, s.Q = (v.to(t).contiguous() for v in (z, torch.maximum(w.expand(ny, nx), z), P, Q))
    return s


def _solver(s):
    g = celeris.Solver(s.z, s.dx, s.dy, s.dt, dtype=s.dtype, model=s.model, g=G, Bd=BD, theta=THETA, eps=s.eps, K=s.K,
                       ws=s.ws, friction=s.friction, fcoef=s.fcoef)
    for side, (kind, width, comps) in s.sides.items():
        g.set_boundary(side, kind, width, comps)
    return g


def _gauges(case, s, n, seed):
    """Cells in water, spread over the grid."""
    rng = random.Random(int(seed) * 31 + 5)
    out = []
    top = {"beach": 0.6, "hump": 0.6, "directional": 0.6, "shoal": 0.98}[case["bed"]]
    for _ in range(n):
        out.append((int(rng.uniform(0.05, top) * s.nx), int(rng.uniform(0.1, 0.9) * s.ny)))
    return out


def _members(case, seed):
    """Uneven sizes up to the case's largest, one scene each."""
    rng = random.Random(int(case["nx"]) * 1000 + case["members"])
    sizes = [(rng.randint(min(128, case["nx"]), case["nx"]), rng.randint(min(128, case["ny"]), case["ny"]))
             for _ in range(case["members"])]
    return [_scene(case, int(seed) * 1009 + k, nx, ny) for k, (nx, ny) in enumerate(sizes)]


RENDER = (dict(mode="fresnel", dry_h=1e-3, zmin=-10.0, zmax=3.0, exaggeration=5.0, view=(0.3, 0.2, -0.8), grid=100.0),
          dict(mode="eta", vmin=-0.4, vmax=0.4, zmin=-10.0, zmax=3.0),
          dict(mode="speed", vmin=0.0, vmax=1.0, zmin=-10.0, zmax=3.0))


# ------------------------------------------------------------------- the path

def prepare(case, seed):
    if case["task"] == "ensemble":
        scenes = _members(case, seed)
        members = [_solver(s) for s in scenes]
        return case, scenes, celeris.Ensemble(members), None
    s = _scene(case, seed)
    g = _solver(s)
    more = None
    if case["task"] == "gauges":
        g.set_gauges(_gauges(case, s, 16, seed), 1, case["steps"])
    if case["task"] == "gradient":
        ij, obs = _observed(case, s, seed)
        size = celeris.adjoint_scratch_bytes(g, case["steps"], 16, case["every"], bed=True)
        more = (ij, obs, torch.empty(size, dtype=torch.uint8, device="cuda"))
    return case, s, g, more


def run(state):
    case, s, g, more = state
    task, n = case["task"], case["steps"]
    if task == "ensemble":
        for m, t in zip(g.members, s):
            m.set_state(t.w, t.P, t.Q)
        g.step(n)
        fields = [m.state() for m in g.members]
        return {k: torch.cat([f[v].reshape(-1) for f in fields]) for v, k in enumerate("wPQ")}
    g.set_state(s.w, s.P, s.Q)
    if task == "frames":
        return [g.render(**RENDER[k % len(RENDER)]) for k in range(n)]
    if task == "gradient":
        ij, obs, scratch = more
        loss, eta, gw, gz = celeris.gauge_misfit_gradient(g, n, ij, obs, case["every"], bed=True, scratch=scratch)
        return {"loss": loss, "eta": eta, "grad_w": gw, "grad_z": gz}
    if task == "runup":
        g.runup_enable(s.delta)
    g.step(n)
    w, P, Q = g.state()
    out = {"w": w, "P": P, "Q": Q}
    if task == "gauges":
        out["eta"] = g.read_gauges(n)
    if task == "runup":
        r = g.runup()
        out["runup"] = torch.where(torch.isfinite(r), r, s.z)
    return out


def work(case):
    es = 4 if case["dtype"] == "f32" else 8
    n = case["nx"] * case["ny"]
    if case["task"] == "ensemble":
        rng = random.Random(int(case["nx"]) * 1000 + case["members"])
        n = sum(rng.randint(min(128, case["nx"]), case["nx"]) * rng.randint(min(128, case["ny"]), case["ny"])
                for _ in range(case["members"]))
    if case["task"] == "frames":   # state and bed in, one pixel out
        return {"bytes": n * (7 * es + case["steps"] * (4 * es + 4)), "flops": 150.0 * n * case["steps"]}
    # per cell and step: w, P, Q, the bed, two history values of each unknown in and out, U*, V* between the passes (25
    # values), and for each corrector iteration the iterate and the bases again (14); fewer in shallow water, whose
    # lines need no solve.  Two Euler steps open every pass.
    K = case["K"]
    values = (25 + 14 * K) if case["model"] == "bsnq" else (19 + 8 * K)
    flops = (430 if case["model"] == "bsnq" else 280) * (K + 1)
    passes = 1
    if case["task"] == "gradient":   # the run, and its reverse of about twice the values and three times the operations
        values, flops, passes = 3 * values, 4 * flops, 1
        if case["every"]:
            values, flops = values * 4 // 3, flops * 5 // 4   # the run once more, from checkpoints
    return {"bytes": float(n * es * (6 + case["steps"] * values * passes)), "flops": float(n * case["steps"] * flops)}


def tolerance(case):
    if case["task"] == "frames":
        return "exact"
    # about four times what single precision shows against 64 bits, in these equations written in plain torch as in the
    # solver: largest where a discharge is a small difference of large terms (the shoal's and the island's cross-tank
    # discharge) or a film thins out (the planar beach); double precision scales by the ratio of the roundings, doubled.
    # Gradients in single precision differ by the branches (limiters, wet cells) that the two states take.
    rel, big = {"shoal": (1e-3, 1.5e-2), "island": (2.5e-5, 8e-4), "planar": (2e-5, 3e-4), "hump": (2e-3, 0.1)}.get(
        case["bed"], (8e-6, 1e-4))
    if case["dtype"] == "f32":
        return {"rel": rel, "max": big}
    if case["task"] == "gradient":
        return {"rel": 1e-13, "max": 4e-12}
    return {"rel": 4e-9 * rel, "max": 4e-9 * big}


# ------------------------------------------------ the same in plain torch, 64 bits

def _pad(v):
    """Two ghost layers mirrored evenly on every side."""
    v = torch.cat([v[:, :2].flip(1), v, v[:, -2:].flip(1)], 1)
    return torch.cat([v[:2].flip(0), v, v[-2:].flip(0)], 0)


def _desing(h, eps):
    h4 = (h * h) * (h * h)
    return math.sqrt(2.0) * h / torch.sqrt(h4 + torch.where(h4 >= eps, h4, torch.full_like(h4, eps)))


def _sqrt(x):
    """A square root whose derivative at 0 is 0."""
    ok = x > 0
    return torch.where(ok, torch.sqrt(torch.where(ok, x, torch.ones_like(x))), torch.zeros_like(x))


def _pos(x):
    return torch.where(x >= 0, x, torch.zeros_like(x))


def _top(a, b):
    return torch.where(a >= b, a, b)


def _low(a, b):
    return torch.where(a <= b, a, b)


class Model:
    """The equations on one scene, in the type of z."""

    def __init__(self, s, z):
        self.s = s
        f = z.dtype
        self.f = f
        zp = _pad(z)
        Bc = 0.25 * (zp[:-1, :-1] + zp[:-1, 1:] + zp[1:, :-1] + zp[1:, 1:])          # corners -1 .. n + 1
        Bb = 0.25 * (Bc[:-1, :-1] + Bc[:-1, 1:] + Bc[1:, :-1] + Bc[1:, 1:])          # cells -1 .. n
        self.Bx = 0.5 * (Bc[1:-2] + Bc[2:-1])      # [ny, nx + 3]: x-faces -1 .. nx + 1 of the rows
        self.By = 0.5 * (Bc[:, 1:-2] + Bc[:, 2:-1])
        self.Bbar = Bb[1:-1, 1:-1]
        dr = s.ws - Bb
        d = torch.where(dr > 0, dr, torch.zeros_like(dr))
        self.d = d[1:-1, 1:-1]
        self.ddx = (d[1:-1, 2:] - d[1:-1, :-2]) / (2.0 * s.dx)
        self.ddy = (d[2:, 1:-1] - d[:-2, 1:-1]) / (2.0 * s.dy)
        self.gam = self._sponge()
        self.bsnq = s.model == celeris.BSNQ
        if self.bsnq:
            self.lines = [self._line(0), self._line(1)]

    def _sponge(self):
        s, f = self.s, self.f
        gam = torch.ones((s.ny, s.nx), dtype=f, device="cuda")
        for side, (kind, width, _) in s.sides.items():
            if kind != celeris.SPONGE or width <= 0:
                continue
            n = s.nx if side in (W, E) else s.ny
            k = torch.arange(n, dtype=torch.float64, device="cuda")
            if side in (E, N):
                k = n - 1 - k
            v = torch.where(k < width, 0.5 * (1.0 + torch.cos(math.pi * (width - k - 0.5) / width)), torch.ones_like(k))
            v = v.to(f)
            gam = torch.minimum(gam, v[None, :] if side in (W, E) else v[:, None])
        return gam

    def _line(self, dirn):
        """Eq. 23's rows of every line, and the factors of their cyclic reduction."""
        s = self.s
        h = s.dx if dirn == 0 else s.dy
        d, da = (self.d, self.ddx) if dirn == 0 else (self.d.T, self.ddy.T)
        r = (BD + 1.0 / 3.0) * d * d / (h * h)
        q = d * da / (6.0 * h)
        a, b, c = q - r, 1.0 + 2.0 * r, -q - r
        full = (a, b, c)
        a0, cn = a[:, :1], c[:, -1:]
        lo, hi = ((W, E), (S, N))[dirn]
        zero = torch.zeros_like(a0)
        b = torch.cat([b[:, :1] - (zero if s.sides[lo][0] == celeris.SINE else a0), b[:, 1:]], 1)
        b = torch.cat([b[:, :-1], b[:, -1:] - (zero if s.sides[hi][0] == celeris.SINE else cn)], 1)
        a = torch.cat([zero, a[:, 1:]], 1)
        c = torch.cat([c[:, :-1], zero], 1)
        steps, k, n = [], 1, a.shape[1]
        while k < n:
            # every row takes k1 times the row k before it and k2 times the row k after it away
            k1 = torch.cat([torch.zeros_like(a[:, :k]), a[:, k:] / b[:, :-k]], 1)
            k2 = torch.cat([c[:, :-k] / b[:, k:], torch.zeros_like(c[:, :k])], 1)
            steps.append((k, k1[:, k:], k2[:, :-k]))
            z = torch.zeros_like(a[:, :k])
            am, cm = torch.cat([z, a[:, :-k]], 1), torch.cat([z, c[:, :-k]], 1)
            ap, cp = torch.cat([a[:, k:], z], 1), torch.cat([c[:, k:], z], 1)
            b = b - cm * k1 - ap * k2
            a, c = -am * k1, -cp * k2
            k *= 2
        return full, steps, b, (a0, cn)

    def _solve(self, dirn, r):
        _, steps, b, _ = self.lines[dirn]
        for k, k1, k2 in steps:
            m = torch.nn.functional.pad(k1 * r[:, :-k], (k, 0))
            p = torch.nn.functional.pad(k2 * r[:, k:], (0, k))
            r = r - m - p
        return r / b

    def makers(self, t):
        """(w, P, Q) of both ghost layers of every maker side at time t."""
        s, out = self.s, {}
        for side, (kind, _, comps) in s.sides.items():
            if kind != celeris.SINE:
                continue
            rows = []
            for layer in range(2):
                if side in (W, E):
                    dadj = self.d[:, 0 if side == W else -1]
                    x = ((-1 - layer if side == W else s.nx + layer) + 0.5) * s.dx
                    x = torch.full((s.ny,), x, dtype=torch.float64, device="cuda")
                    y = (torch.arange(s.ny, dtype=torch.float64, device="cuda") + 0.5) * s.dy
                else:
                    raise ValueError("makers stand on the west or east side here")
                dadj = dadj.double()
                wet = dadj > 0
                safe = torch.where(wet, dadj, torch.ones_like(dadj))
                eta, Pg, Qg = (torch.zeros_like(x) for _ in range(3))
                for amp, T, th, ph in comps:
                    om = 2.0 * math.pi / T
                    k0 = om * om / G
                    k = k0 / torch.sqrt(torch.tanh(k0 * safe))
                    e = amp * torch.sin(om * t - k * math.cos(th) * x - k * math.sin(th) * y + ph)
                    e = torch.where(wet, e, torch.zeros_like(e))
                    eta, Pg, Qg = eta + e, Pg + om / k * math.cos(th) * e, Qg + om / k * math.sin(th) * e
                rows.append([(v.to(self.f))[:, None] for v in (s.ws + eta, Pg, Qg)])
            out[side] = rows
        return out

    def ghosts(self, w, P, Q, mk):
        def side(k, v, sgn, var):
            if k in mk:
                a, b = mk[k][0][var], mk[k][1][var]
                return [b, a] if k == W else [a, b]
            return [sgn * (v[:, :2] if k == W else v[:, -2:]).flip(1)]

        ext = []
        for var, (v, sx, sy) in enumerate(((w, 1.0, 1.0), (P, -1.0, 1.0), (Q, 1.0, -1.0))):
            v = torch.cat(side(W, v, sx, var) + [v] + side(E, v, sx, var), 1)
            ext.append(torch.cat([sy * v[:2].flip(0), v, sy * v[-2:].flip(0)], 0))
        return ext

    def _flux(self, q, B, normal):
        """Fluxes through faces 0 .. n along the last axis; q: (w, P, Q) with two ghost layers there."""
        lo, hi = [], []
        for v in q:
            qm, q0, qp = v[:, :-2], v[:, 1:-1], v[:, 2:]
            a, b, c = THETA * (q0 - qm), 0.5 * (qp - qm), THETA * (qp - q0)
            up, dn = _low(a, _low(b, c)), _top(a, _top(b, c))
            sl = torch.where(up > 0, up, torch.where(dn < 0, dn, torch.zeros_like(dn)))
            lo.append(q0 - 0.5 * sl)
            hi.append(q0 + 0.5 * sl)
        w0, Blo, Bhi = q[0][:, 1:-1], B[:, :-1], B[:, 1:]
        up = hi[0] < Bhi
        dn = (~up) & (lo[0] < Blo)
        lo[0], hi[0] = (torch.where(up, 2.0 * w0 - Bhi, torch.where(dn, Blo, lo[0])),
                        torch.where(up, Bhi, torch.where(dn, 2.0 * w0 - Blo, hi[0])))
        t = 3 - normal
        Bf = B[:, 1:-1]
        wL, nL, tL = hi[0][:, :-1], hi[normal][:, :-1], hi[t][:, :-1]
        wR, nR, tR = lo[0][:, 1:], lo[normal][:, 1:], lo[t][:, 1:]
        hL, hR = _pos(wL - Bf), _pos(wR - Bf)
        kL, kR = _desing(hL, self.s.eps), _desing(hR, self.s.eps)
        uL, vL, uR, vR = kL * nL, kL * tL, kR * nR, kR * tR
        qL, sL, qR, sR = hL * uL, hL * vL, hR * uR, hR * vR
        cL, cR = _sqrt(G * hL), _sqrt(G * hR)
        ap = _pos(_top(uL + cL, uR + cR))
        am = -_pos(-_low(uL - cL, uR - cR))
        den = ap - am
        ok = den > 0
        den = torch.where(ok, den, torch.ones_like(den))
        H = ((ap * qL - am * qR + ap * am * (wR - wL)) / den,
             (ap * (qL * uL + 0.5 * G * hL * hL) - am * (qR * uR + 0.5 * G * hR * hR) + ap * am * (qR - qL)) / den,
             (ap * qL * vL - am * qR * vR + ap * am * (sR - sL)) / den)
        H = [torch.where(ok, h, torch.zeros_like(h)) for h in H]
        return H if normal == 1 else [H[0], H[2], H[1]]

    def rhs(self, w, P, Q, mk):
        """E, F, G, F*, G* (Eq. 9-13, 31-32)."""
        s = self.s
        dx, dy = s.dx, s.dy
        X = self.ghosts(w, P, Q, mk)
        Hx = self._flux([v[2:-2] for v in X], self.Bx, 1)
        Hy = [h.T for h in self._flux([v[:, 2:-2].T for v in X], self.By.T, 2)]
        div = [-(hx[:, 1:] - hx[:, :-1]) / dx - (hy[1:] - hy[:-1]) / dy for hx, hy in zip(Hx, Hy)]
        hb = w - self.Bbar
        E_ = div[0]
        F = div[1] - G * hb * (self.Bx[:, 2:-1] - self.Bx[:, 1:-2]) / dx
        Gq = div[2] - G * hb * (self.By[2:-1] - self.By[1:-2]) / dy
        if s.friction != celeris.FRIC_NONE:
            k = _desing(_pos(hb), s.eps)
            fc = s.fcoef
            if s.friction == celeris.FRIC_MANNING:
                pos = k > 0
                fc = G * s.fcoef ** 2 * torch.where(pos, torch.where(pos, k, torch.ones_like(k)) ** (1.0 / 3.0),
                                                    torch.zeros_like(k))
            m = fc * _sqrt(P * P + Q * Q) * k * k
            F = F - m * P
            Gq = Gq - m * Q
        if not self.bsnq:
            z = torch.zeros_like(w)
            return E_, F, Gq, z, z

        def at(v, i, j):
            return v[2 + j:v.shape[0] - 2 + j, 2 + i:v.shape[1] - 2 + i]

        e, Pe, Qe = X
        c = w
        exx = (at(e, 1, 0) - 2.0 * c + at(e, -1, 0)) / dx ** 2
        eyy = (at(e, 0, 1) - 2.0 * c + at(e, 0, -1)) / dy ** 2
        exy = (at(e, 1, 1) - at(e, 1, -1) - at(e, -1, 1) + at(e, -1, -1)) / (4.0 * dx * dy)
        exxx = (at(e, 2, 0) - 2.0 * at(e, 1, 0) + 2.0 * at(e, -1, 0) - at(e, -2, 0)) / (2.0 * dx ** 3)
        eyyy = (at(e, 0, 2) - 2.0 * at(e, 0, 1) + 2.0 * at(e, 0, -1) - at(e, 0, -2)) / (2.0 * dy ** 3)
        exyy = ((at(e, 1, 1) - 2.0 * at(e, 1, 0) + at(e, 1, -1))
                - (at(e, -1, 1) - 2.0 * at(e, -1, 0) + at(e, -1, -1))) / (2.0 * dx * dy * dy)
        exxy = ((at(e, 1, 1) - 2.0 * at(e, 0, 1) + at(e, -1, 1))
                - (at(e, 1, -1) - 2.0 * at(e, 0, -1) + at(e, -1, -1))) / (2.0 * dx * dx * dy)
        d, ax, ay = self.d, self.ddx, self.ddy
        F = F + BD * G * d ** 3 * (exxx + exyy) + BD * G * d * d * (ax * (2.0 * exx + eyy) + ay * exy)
        Gq = Gq + BD * G * d ** 3 * (eyyy + exxy) + BD * G * d * d * (ay * (2.0 * eyy + exx) + ax * exy)

        def first(v):
            vx, vy = (at(v, 1, 0) - at(v, -1, 0)) / (2.0 * dx), (at(v, 0, 1) - at(v, 0, -1)) / (2.0 * dy)
            return vx, vy, (at(v, 1, 1) - at(v, 1, -1) - at(v, -1, 1) + at(v, -1, -1)) / (4.0 * dx * dy)

        Qx, Qy, Qxy = first(Qe)
        Px, Py, Pxy = first(Pe)
        B3 = BD + 1.0 / 3.0
        Fs = d * ax * Qy / 6.0 + d * ay * Qx / 6.0 + B3 * d * d * Qxy
        Gs = d * ay * Px / 6.0 + d * ax * Py / 6.0 + B3 * d * d * Pxy
        return E_, F, Gq, Fs, Gs

    def _new(self, dirn, base, inc, mk0, mk1):
        """P (or Q) at the new time: the increment solves Eq. 21 (22), the makers' ghost increments known."""
        if not self.bsnq:
            return base + inc
        if dirn == 1:
            base, inc = base.T, inc.T
        a0, cn = self.lines[dirn][3]
        lo, hi = ((W, E), (S, N))[dirn]
        if lo in mk1:
            inc = torch.cat([inc[:, :1] - a0 * (mk1[lo][0][1 + dirn] - mk0[lo][0][1 + dirn]), inc[:, 1:]], 1)
        if hi in mk1:
            inc = torch.cat([inc[:, :-1], inc[:, -1:] - cn * (mk1[hi][0][1 + dirn] - mk0[hi][0][1 + dirn])], 1)
        x = base + self._solve(dirn, inc)
        return x.T if dirn == 1 else x

    def clamp(self, w):
        return torch.where(w <= self.Bbar, self.Bbar, w)

    def step(self, n, w, P, Q, h1, h2, t0):
        """Step n of a fresh history from time t0; h1, h2: the right sides of the two steps before it."""
        s, dt = self.s, self.s.dt
        mk0, mk1 = self.makers(t0), self.makers(t0 + dt)
        R = self.rhs(w, P, Q, mk0)
        if n < 2:
            inc = [dt * r for r in R[:3]]
            if n == 1:
                inc[1], inc[2] = inc[1] + (R[3] - h1[3]), inc[2] + (R[4] - h1[4])
        else:
            inc = [dt / 12.0 * (23.0 * r - 16.0 * a + 5.0 * b) for r, a, b in zip(R[:3], h1, h2)]
            for v in (1, 2):
                inc[v] = inc[v] + 2.0 * R[v + 2] - 3.0 * h1[v + 2] + h2[v + 2]
        last = s.K if n >= 2 else 0
        for stage in range(last + 1):
            if stage:
                C = self.rhs(w1, P1, Q1, mk1)
                inc = [dt / 24.0 * (9.0 * c + 19.0 * r - 5.0 * a + b) for c, r, a, b in zip(C[:3], R, h1, h2)]
                for v in (1, 2):
                    inc[v] = inc[v] + C[v + 2] - R[v + 2]
            w1 = self.clamp(w + inc[0])
            P1 = self._new(0, P, inc[1], mk0, mk1)
            Q1 = self._new(1, Q, inc[2], mk0, mk1)
            if stage == last:
                w1 = torch.where((self.gam < 1.0) & (self.d > 0), s.ws + self.gam * (w1 - s.ws), w1)
                P1, Q1 = P1 * self.gam, Q1 * self.gam
            wet = w1 - self.Bbar > 0
            P1, Q1 = (torch.where(wet, v, torch.zeros_like(v)) for v in (P1, Q1))
        return (w1, P1, Q1) + R

    def start(self, w, P, Q):
        w = self.clamp(w)
        wet = w - self.Bbar > 0
        return w, torch.where(wet, P, torch.zeros_like(P)), torch.where(wet, Q, torch.zeros_like(Q))


def _fields(case, s, f=torch.float64):
    with torch.no_grad():
        m = Model(s, s.z.to(f))
        w, P, Q = m.start(s.w.to(f), s.P.to(f), s.Q.to(f))
        zero = [torch.zeros_like(w)] * 5
        h1, h2, eta, top = zero, zero, [], None
        if case["task"] == "gauges":
            ij = torch.tensor(_gauges(case, s, 16, s.seed), device="cuda")
        if case["task"] == "runup":
            low = torch.full_like(w, -math.inf)
            top = torch.where(w - m.Bbar > s.delta, w, low)
        for n in range(case["steps"]):
            out = m.step(n, w, P, Q, h1, h2, n * s.dt)
            w, P, Q = out[:3]
            h1, h2 = list(out[3:]), h1
            if case["task"] == "gauges":
                eta.append(w[ij[:, 1], ij[:, 0]] - s.ws)
            if top is not None:
                top = torch.where(w - m.Bbar > s.delta, torch.maximum(top, w), top)
        out = {"w": w, "P": P, "Q": Q}
        if eta:
            out["eta"] = torch.stack(eta).cpu().numpy()
        if top is not None:
            out["runup"] = torch.where(torch.isfinite(top), top, s.z.to(f))
    return out


def _gradients(case, s, seed, f=torch.float64):
    ij, obs = _observed(case, s, seed)
    z = s.z.to(f).requires_grad_(True)
    m = Model(s, z)
    w, P, Q = m.start(s.w.to(f), s.P.to(f), s.Q.to(f))
    w0 = w
    w0.retain_grad()
    zero = [torch.zeros_like(w)] * 5
    h1, h2, eta = zero, zero, []
    k = torch.tensor(ij, device="cuda")
    for n in range(case["steps"]):
        def one(w, P, Q, *h, n=n):
            return m.step(n, w, P, Q, h[:5], h[5:], n * s.dt)
        out = checkpoint(one, w, P, Q, *h1, *h2, use_reentrant=False)
        w, P, Q = out[:3]
        h1, h2 = list(out[3:]), h1
        eta.append(w[k[:, 1], k[:, 0]] - s.ws)
    eta = torch.stack(eta)
    loss = 0.5 * ((eta - obs.to(f)) ** 2).sum()
    loss.backward()
    return {"loss": float(loss.detach()), "eta": eta.detach(), "grad_w": w0.grad, "grad_z": z.grad}


def _observed(case, s, seed):
    """Gauges, and records there of another wave field: what the misfit compares with."""
    gen = torch.Generator(device="cpu").manual_seed(int(seed))
    obs = (0.2 * torch.rand((case["steps"], 16), generator=gen, dtype=torch.float64) - 0.1).to(s.dtype).cuda()
    return _gauges(case, s, 16, seed), obs


def exact(case, seed, f=torch.float64):
    if case["task"] == "frames":   # bytes, compared as they are
        return None
    if case["task"] == "ensemble":
        parts = [_fields(case, s, f) for s in _members(case, seed)]
        return {k: torch.cat([p[k].reshape(-1) for p in parts]) for k in "wPQ"}
    s = _scene(case, seed)
    s.seed = seed
    return _gradients(case, s, seed, f) if case["task"] == "gradient" else _fields(case, s, f)
