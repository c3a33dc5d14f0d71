"""Timed cases of the lattice library: whole calls a user's program makes.

A pass advances a lattice (or a batch of lattices) by the number of time steps
between two snapshots and reads the snapshot: c1, c2, the velocity and the
pressure, which are what post-processing and a restart need.  Snapshots of
FP64 lattices stay FP64; those of the reduced storages are kept in FP32.
"""
import math
import random

import numpy as np
import torch

import paper_1710_09534_gb300 as tlbm

PERIODIC, WETTING, NEUTRAL, LID = 0, 1, 2, 3
NAMES = ("c1", "c2", "ux", "uy", "p")
NAMES3 = ("c1", "c2", "ux", "uy", "uz", "p")


def listed():
    flat = dict(collision="bgk", inplace=False)
    return [
        # two drops on a wetting wall, the smallest lattice users run: launches and latency
        dict(flat, name="drops_128x64_fp64", problem="drops", nx=128, ny=64, storage="fp64", steps=500),
        # a compound drop hitting a cylinder at the paper's size, density ratio 10
        dict(flat, name="impact_240x280_fp64", problem="impact", nx=240, ny=280, storage="fp64", steps=200),
        # a compound drop sheared by a moving lid, between two snapshots of a 20000-step run
        dict(flat, name="shear_512x256_fp32", problem="shear", nx=512, ny=256, storage="fp32", steps=300),
        # the large lattice of drops on a wall and in the bulk, in each storage
        dict(flat, name="drops_2048x2048_fp64", problem="drops", nx=2048, ny=2048, storage="fp64", steps=50),
        dict(flat, name="drops_2048x2048_fp32", problem="drops", nx=2048, ny=2048, storage="fp32", steps=100),
        dict(flat, name="drops_2048x2048_fp16", problem="drops", nx=2048, ny=2048, storage="fp16", steps=100),
        # the impact at full size: solid nodes and the density-contrast update
        dict(flat, name="impact_1024x2048_fp32", problem="impact", nx=1024, ny=2048, storage="fp32", steps=100),
        # the multiple-relaxation-time collision on an odd-sized lattice
        dict(name="drops_777x501_fp64_mrt", problem="drops", nx=777, ny=501, storage="fp64", collision="mrt",
             inplace=False, steps=50),
        # in-place streaming, chosen where memory is short; an odd step count ends on the in-place swap
        dict(name="drops_2048x1024_fp32_inplace", problem="drops", nx=2048, ny=1024, storage="fp32", collision="bgk",
             inplace=True, steps=101),
        # many independent lattices of mixed sizes advanced together, as the server does
        dict(name="batch_32_fp32", problem="batch", count=32, lo=64, hi=512, storage="fp32", steps=100),
        # three-dimensional drops on a wall
        dict(name="drops3d_192x96x192_fp32", problem="drops3d", nx=192, ny=96, nz=192, storage="fp32", steps=600),
        dict(name="drops3d_96x64x80_fp64", problem="drops3d", nx=96, ny=64, nz=80, storage="fp64", steps=200),
    ]


# rough nanoseconds per node update, to keep a drawn case within the largest listed one
_NS = {"fp64": 0.6, "fp32": 0.07, "fp16": 0.05, "bf16": 0.05}


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.6 else -(-n // 32) * 32

    problem = rng.choice(["drops", "drops", "drops", "impact", "shear", "batch", "drops3d"])
    storage = rng.choice(["fp64", "fp32", "fp32", "fp16", "bf16"])
    if problem == "batch":
        count, hi = rng.randint(8, 32), size(128, 512)
        case = dict(problem=problem, count=count, lo=64, hi=hi, storage=rng.choice(["fp32", "fp16", "fp64"]))
        nodes = sum(n * n for n in _sides(case))
    elif problem == "drops3d":
        case = dict(problem=problem, nx=size(32, 192), ny=size(24, 96), nz=size(32, 192),
                    storage=rng.choice(["fp64", "fp32"]))
        nodes = 2 * case["nx"] * case["ny"] * case["nz"]
    else:
        lo, hi = (96, 2048) if problem == "drops" else (160, 1024)
        nx = size(lo, hi)
        ny = size(lo, hi) if problem != "impact" else max(nx, size(lo, hi))
        mrt = problem != "shear" and rng.random() < 0.25
        case = dict(problem=problem, nx=nx, ny=ny, storage=storage, collision="mrt" if mrt else "bgk",
                    inplace=problem == "drops" and not mrt and rng.random() < 0.3)
        nodes = nx * ny * (4 if mrt else 1)
    most = 70e6 / (nodes * _NS[case["storage"]])
    case["steps"] = max(9, min(rng.randint(60, 400), int(most)))
    return case


def _sides(case):
    r = random.Random("%d %d %d" % (case["count"], case["lo"], case["hi"]))
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    return [max(case["lo"], int(round(math.exp(r.uniform(lo, hi)) / 8)) * 8) for _ in range(case["count"])]


# ---- inputs ------------------------------------------------------------------

def _profile(grid, centre, radius, sizes, periodic, width=4.0):
    """0.5 + 0.5 tanh(2 (R - r) / D) around `centre` (minimum image on periodic axes)."""
    r2 = 0.0
    for x, c, n, per in zip(grid, centre, sizes, periodic):
        d = x - c
        if per:
            d = (d + n / 2) % n - n / 2
        r2 = r2 + d * d
    return 0.5 + 0.5 * torch.tanh(2.0 * (radius - torch.sqrt(r2)) / width)


def _params(sigma=1e-3, theta=(60.0, 90.0, 120.0), rho=(1.0, 1.0, 1.0), nu=(0.1, 0.1, 0.1), mobility=0.1, lid_u=0.0,
            sigma12=None, mrt=False):
    s12 = sigma if sigma12 is None else sigma12
    return dict(sigma12=s12, sigma13=sigma, sigma23=sigma, theta12_deg=theta[0], theta13_deg=theta[1],
                theta23_deg=theta[2], rho1=rho[0], rho2=rho[1], rho3=rho[2], nu1=nu[0], nu2=nu[1], nu3=nu[2],
                M0=mobility * s12, D=4.0, tau1=0.8, tau2=0.8, gx=0.0, gy=0.0, lid_u=lid_u,
                collision=1.0 if mrt else 0.0, mrt_s_f=1.2 if mrt else 1.0, mrt_s_g=1.3 if mrt else 1.0)


def _theta12(s12, s13, s23, t13, t23):
    c = (s13 * math.cos(math.radians(t13)) - s23 * math.cos(math.radians(t23))) / s12
    return math.degrees(math.acos(c))


def _free(rng, lo, hi):
    return lo + (hi - lo) * rng.random()


def _drops(nx, ny, rng, dev):
    """Drops of fluids 1 and 2 every 40 nodes on the wetting bottom wall, compound drops in the bulk, in a slow stream."""
    c1 = torch.zeros(ny, nx, dtype=torch.float64, device=dev)
    c2 = torch.zeros_like(c1)
    ay = torch.arange(ny, dtype=torch.float64, device=dev)[:, None]
    ax = torch.arange(nx, dtype=torch.float64, device=dev)[None, :]

    # the wall drops come in groups whose drops do not overlap: one profile of the nearest one serves all of them
    pitch = nx / max(1, nx // 40)
    shift = _free(rng, 0, pitch)
    h = min(ny, 64)
    near = torch.floor((ax - shift) / pitch)
    centre = shift + (near + 0.5) * pitch
    prof = 0.5 + 0.5 * torch.tanh(2.0 * (_free(rng, 14, 17) - torch.sqrt((ax - centre) ** 2 + (ay[:h] + 0.5) ** 2)) / 4.0)
    first = (near % 2 == 0).to(torch.float64)
    c1[:h] = prof * first
    c2[:h] = prof * (1 - first)
    if ny > 140:
        rows = max(1, (ny - 100) // 90)
        for j in range(rows):
            for xc in np.arange(45.0, nx - 20, 180.0):
                radius = _free(rng, 10, 24)
                x, y = xc + _free(rng, -20, 20), 90 + 90.0 * j + _free(rng, -10, 10)
                if y + radius + 12 < ny:
                    y0, y1 = int(y - radius - 30), min(ny, int(y + radius + 31))
                    x0, x1 = max(0, int(x - radius - 30)), min(nx, int(x + radius + 31))
                    win = (ax[:, x0:x1], ay[y0:y1])
                    shell = _profile(win, (x, y), radius, (nx, ny), (False, False))
                    core = _profile(win, (x, y), 0.55 * radius, (nx, ny), (False, False))
                    keep = (c1[y0:y1, x0:x1] + c2[y0:y1, x0:x1]) < 1e-9
                    c1[y0:y1, x0:x1] = torch.where(keep, core, c1[y0:y1, x0:x1])
                    c2[y0:y1, x0:x1] = torch.where(keep, shell - core, c2[y0:y1, x0:x1])
    ux = 5e-4 * torch.sin(2 * math.pi * (ay + 0.5) / ny) + torch.zeros_like(c1)
    return c1, c2, ux, torch.zeros_like(c1)


def _problem2(case, seed, dev):
    """Edges, mask, parameters and initial fields of a two-dimensional problem."""
    rng = random.Random(int(seed) * 7919 + 13)
    nx, ny, mrt = case["nx"], case["ny"], case["collision"] == "mrt"
    ay = torch.arange(ny, dtype=torch.float64, device=dev)[:, None]
    ax = torch.arange(nx, dtype=torch.float64, device=dev)[None, :]
    mask = torch.zeros(ny, nx, dtype=torch.uint8, device=dev)
    if case["problem"] == "drops":
        return ((PERIODIC, PERIODIC, WETTING, NEUTRAL), mask, _params(mrt=mrt)) + _drops(nx, ny, rng, dev)
    if case["problem"] == "shear":
        u0 = 0.01
        r = min(nx, 2 * ny) / 512.0
        xc = nx / 2 + _free(rng, -nx / 8, nx / 8)
        core = _profile((ax, ay), (xc, -0.5), 30 * r * _free(rng, 0.9, 1.1), (nx, ny), (True, False))
        c2 = _profile((ax, ay), (xc, -0.5), 50 * r * _free(rng, 0.95, 1.1), (nx, ny), (True, False)) - core
        ux = torch.zeros_like(core)
        ux[ny - 1] = u0
        par = _params(theta=(_theta12(2e-3, 1e-3, 1e-3, 90.0, 135.0), 90.0, 135.0), rho=(1.0, 2.0, 1.0),
                      nu=(0.05, 0.1, 0.05), lid_u=u0, sigma12=2e-3, mobility=0.1)
        return (PERIODIC, PERIODIC, WETTING, LID), mask, par, core, c2, ux, torch.zeros_like(ux)
    # impact: a compound drop falling onto a wetting cylinder, fully periodic
    size = min(nx, ny)
    cyl, shell = size / 8.5, size / 10.0
    mask = (((ax - nx / 2) ** 2 + (ay - size / 2) ** 2) <= cyl * cyl).to(torch.uint8)
    at = (nx / 2 + _free(rng, -4, 4), size / 2 + cyl + shell + _free(rng, 6, 12))
    c1 = _profile((ax, ay), at, 0.55 * shell, (nx, ny), (True, True))
    c2 = _profile((ax, ay), at, shell, (nx, ny), (True, True)) - c1
    c1, c2 = c1 * (mask == 0), c2 * (mask == 0)
    speed = math.sqrt(10.0 * 0.01 / (10.0 * 2.0 * shell))
    par = _params(sigma=0.01, theta=(90.0, 60.0, 60.0), rho=(10.0, 10.0, 1.0), nu=(0.02, 0.02, 0.02), mobility=0.1,
                  mrt=mrt)
    return (PERIODIC,) * 4, mask, par, c1, c2, torch.zeros_like(c1), -speed * (c1 + c2)


def _problem3(case, seed, dev):
    rng = random.Random(int(seed) * 7919 + 13)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    grid = (torch.arange(nx, dtype=torch.float64, device=dev)[None, None, :],
            torch.arange(ny, dtype=torch.float64, device=dev)[None, :, None],
            torch.arange(nz, dtype=torch.float64, device=dev)[:, None, None])
    c = [torch.zeros(nz, ny, nx, dtype=torch.float64, device=dev) for _ in range(2)]
    radius = min(16.0, 0.3 * min(nx, ny, nz))
    sx, sz = _free(rng, 0, nx), _free(rng, 0, nz)
    mx, mz = max(1, int(nx // (2.5 * radius))), max(1, int(nz // (2.5 * radius)))
    for j in range(mz):
        for i in range(mx):
            at = ((sx + i * nx / mx) % nx, -0.5, (sz + j * nz / mz) % nz)
            p = _profile(grid, at, radius * _free(rng, 0.9, 1.0), (nx, ny, nz), (True, False, True))
            c[(i + j) % 2] = torch.maximum(c[(i + j) % 2], p)
    z = torch.zeros_like(c[0])
    edges = (PERIODIC, PERIODIC, WETTING, NEUTRAL, PERIODIC, PERIODIC)
    return edges, torch.zeros(nz, ny, nx, dtype=torch.uint8, device=dev), _params(), c[0], c[1], z, z, z


def _members(case, seed):
    """The batch's lattices as single problems, one seed each."""
    return [(dict(problem="drops", nx=n, ny=n, collision="bgk"), int(seed) * 1000 + i)
            for i, n in enumerate(_sides(case))]


def _lattice(case, seed, storage, inplace, stream, dev):
    edges, mask, par, c1, c2, ux, uy = _problem2(case, seed, dev)
    lat = tlbm.Lattice(case["nx"], case["ny"], storage, edges, stream=stream, inplace=inplace)
    lat.set_geometry(mask.cpu().numpy())
    lat.set_params(par)
    torch.cuda.synchronize()
    lat.set_fields_device(c1, c2, ux, uy)
    torch.cuda.synchronize()
    out = torch.empty(len(NAMES), case["ny"], case["nx"], dtype=torch.float64, device=dev)
    return lat, out


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    if case["problem"] == "drops3d":
        edges, mask, par, c1, c2, ux, uy, uz = _problem3(case, seed, dev)
        lat = tlbm.Lattice3D(case["nx"], case["ny"], case["nz"], edges, precision=case["storage"])
        lat.set_geometry(mask.cpu().numpy())
        lat.set_params(par)
        lat.set_fields(*(a.cpu().numpy() for a in (c1, c2, ux, uy, uz)))
        return dict(case=case, lat=lat)
    if case["problem"] == "batch":
        members = _members(case, seed)
        tiles = sum(tlbm.Batch.tiles_needed(c["nx"], c["ny"]) for c, _ in members)
        walls = sum(8 * c["nx"] for c, _ in members)
        batch = tlbm.Batch(case["storage"], len(members), tiles, walls)
        # the shape the server starts with
        batch.config(threads=64, rows_small=8, rows_large=32, small_ny=128)
        lats = [_lattice(c, s, case["storage"], False, batch.stream, dev) for c, s in members]
        for lat, _ in lats:
            batch.add(lat)
        return dict(case=case, batch=batch, lats=lats)
    lat, out = _lattice(case, seed, case["storage"], case["inplace"], None, dev)
    return dict(case=case, lat=lat, out=out)


def run(state):
    case = state["case"]
    if case["problem"] == "drops3d":
        state["lat"].step(case["steps"])
        got = state["lat"].fields(NAMES3)
        kind = np.float64 if case["storage"] == "fp64" else np.float32
        return [got[k].astype(kind, copy=False) for k in NAMES3]
    if case["problem"] == "batch":
        batch = state["batch"]
        batch.step(case["steps"])
        with torch.cuda.stream(batch.stream):
            got = []
            for lat, out in state["lats"]:
                lat.fields_device(out, NAMES)
                out = out if case["storage"] == "fp64" else out.to(torch.float32)
                got.append([out[:2], out[2:]])
        return got
    state["lat"].step(case["steps"])
    state["lat"].fields_device(state["out"], NAMES)
    out = state["out"] if case["storage"] == "fp64" else state["out"].to(torch.float32)
    return list(out)


def work(case):
    if case["problem"] == "batch":
        nodes = sum(n * n for n in _sides(case))
    else:
        nodes = case["nx"] * case["ny"] * case.get("nz", 1)
    dims, q = (3, 19) if case["problem"] == "drops3d" else (2, 9)
    dist = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case["storage"]]
    wide = 8 if case["storage"] == "fp64" else 4
    # each step reads and writes the 3 q populations and the c_i u of two components
    step = 2 * (3 * q * dist + 2 * dims * wide)
    # multiplications and additions of the collision, moments and stencils as the equations state them
    flops = (500 if dims == 3 else 310) + (90 if case["problem"] in ("impact", "shear") else 0)
    return {"bytes": nodes * (case["steps"] * step + (3 + dims) * wide), "flops": nodes * case["steps"] * flops}


# ---- the same passes in plain FP64 tensors -------------------------------------

def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["problem"] == "batch":
        got = []
        for i, (c, s) in enumerate(_members(case, seed)):
            a = torch.stack(_Plain(2, *_problem2(c, s, dev)).run(case["steps"])) if i < 8 else None
            got.append(None if a is None else [a[:2], a[2:]])
        return got
    if case["problem"] == "drops3d":
        return _Plain(3, *_problem3(case, seed, dev)).run(case["steps"])
    if case["problem"] != "drops" and case["storage"] in ("fp16", "bf16"):
        return None  # the pressure of a fast, dense drop is within the rounding of 16-bit populations
    return _Plain(2, *_problem2(case, seed, dev)).run(case["steps"])


E2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
E3 = [(0, 0, 0)] + [e for a in range(3) for e in [tuple(s if b == a else 0 for b in range(3)) for s in (1, -1)]] + [
    (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1),
    (0, -1, -1), (0, 1, -1), (0, -1, 1)]
FLUID, TOP, WET, PLAIN, VOID = 0, 1, 2, 3, 4


class _Plain:
    """The model of arXiv:1710.09534, Sec. II, one tensor operation per term."""

    def __init__(self, dims, edges, mask, par, c1, c2, *u):
        self.d, self.p = dims, par
        self.e = E2 if dims == 2 else E3
        rest, axis = (4 / 9, 1 / 9) if dims == 2 else (1 / 3, 1 / 18)
        self.w = [rest if not any(e) else axis if sum(map(abs, e)) == 1 else 1 / 36 for e in self.e]
        self.opp = [self.e.index(tuple(-x for x in e)) for e in self.e]
        kind = torch.where(mask == 1, WET, torch.where(mask == 2, PLAIN, FLUID)).to(torch.uint8)
        self.lid = dims == 2 and edges[3] == LID
        if self.lid:
            kind[-1] = torch.where(kind[-1] == FLUID, TOP, kind[-1])
        self.kind = kind
        self.fluid, self.live = kind == FLUID, kind <= TOP
        self.open, self.wet, self.solid = [], [], []
        for e in self.e:
            k = self.at(kind, e).clone()
            for a in reversed(range(dims)):  # the x edge decides at a corner
                if e[a] and edges[2 * a] != PERIODIC:
                    edge = edges[2 * a + (1 if e[a] > 0 else 0)]
                    k.select(dims - 1 - a, -1 if e[a] > 0 else 0).fill_({WETTING: WET, NEUTRAL: PLAIN, LID: VOID}[edge])
            self.open.append(k <= TOP)
            self.wet.append(k == WET)
            self.solid.append((k == WET) | (k == PLAIN))
        s12, s13, s23 = par["sigma12"], par["sigma13"], par["sigma23"]
        self.lam = (s12 + s13 - s23, s12 + s23 - s13, s13 + s23 - s12)
        l1, l2, l3 = self.lam
        den = l1 * l2 + l1 * l3 + l2 * l3
        self.lam_t = 3 * l1 * l2 * l3 / den if den else 0.0
        self.tau = (par["tau1"], par["tau2"])
        self.mob = [par["M0"] / self.lam[i] for i in range(2)]
        self.eta = [self.mob[i] * 3 / (self.tau[i] - 0.5) for i in range(2)]
        zero = torch.zeros_like(c1)
        self.c = [torch.where(self.fluid, c, zero) for c in (c1, c2)]
        self.lower(self.c)
        self.potentials()
        u = [torch.where(self.live, a, zero) for a in u]
        rho = self.density()
        self.f = [[self.live * self.feq(i, k, self.c[i], self.mu[i], u) for k in range(len(self.e))] for i in range(2)]
        self.g = [self.live * self.geq(k, zero, rho, u) for k in range(len(self.e))]
        self.cu = [[c * a for a in u] for c in self.c]

    def at(self, a, e):
        """a at x + e, wrapped."""
        s = tuple(-x for x in reversed(e))
        return torch.roll(a, s, tuple(range(self.d))) if any(e) else a

    def lower(self, fields):
        """The lid row takes the values of the row below it."""
        if self.lid:
            for a in fields:
                a[-1] = torch.where(self.kind[-1] == TOP, a[-2], a[-1])

    def near(self, a, k):
        """a at x + e_k, the node's own value across a link into a solid."""
        return torch.where(self.open[k], self.at(a, self.e[k]), a)

    def grad(self, a):
        g = [torch.zeros_like(a) for _ in range(self.d)]
        for k in range(1, len(self.e)):
            v = self.near(a, k)
            for b in range(self.d):
                if self.e[k][b]:
                    g[b] += 3 * self.w[k] * self.e[k][b] * v
        return g

    def lap(self, a, ghost=None):
        s = torch.zeros_like(a)
        for k in range(1, len(self.e)):
            v = self.near(a, k) - a
            if ghost is not None:
                v = torch.where(self.wet[k], ghost, v)
            s += 6 * self.w[k] * v
        return s

    def density(self):
        p, (a, b) = self.p, self.c
        return a * p["rho1"] + b * p["rho2"] + (1 - a - b) * p["rho3"]

    def potentials(self):
        p, (a, b) = self.p, self.c
        c3 = 1 - a - b
        cos12, cos13, cos23 = (math.cos(math.radians(p[k])) for k in ("theta12_deg", "theta13_deg", "theta23_deg"))
        ghosts = [4 / p["D"] * (cos13 * a * c3 + cos12 * a * b), 4 / p["D"] * (-cos12 * a * b + cos23 * b * c3)]
        self.mu = []
        for i, c in enumerate((a, b)):
            bulk = self.lam[i] * c * (1 - c) * (1 - 2 * c) - 2 * self.lam_t * a * b * c3
            mu = 12 / p["D"] * bulk - 0.75 * p["D"] * self.lam[i] * self.lap(c, ghosts[i])
            self.mu.append(torch.where(self.fluid, mu, 0.0))
        self.lower(self.mu)

    def dot(self, k, v):
        return sum(self.e[k][b] * v[b] for b in range(self.d) if self.e[k][b]) if any(self.e[k]) else torch.zeros_like(v[0])

    def sk(self, k, u):
        eu = self.dot(k, u)
        return self.w[k] * (3 * eu + 4.5 * eu * eu - 1.5 * sum(x * x for x in u))

    def feq(self, i, k, c, mu, u):
        if k == 0:
            return c + (self.w[0] - 1) * self.eta[i] * mu
        return self.w[k] * (self.eta[i] * mu + 3 * c * self.dot(k, u))

    def geq(self, k, pr, rho, u):
        return 3 * pr * (self.w[k] - (k == 0)) + rho * self.sk(k, u)

    def macros(self):
        p = self.p
        self.c = [torch.where(self.fluid, sum(f), 0.0) for f in self.f]
        self.lower(self.c)
        self.potentials()
        self.rho = self.density()
        m3 = -self.lam[2] * (self.mu[0] / self.lam[0] + self.mu[1] / self.lam[1])
        g1, g2 = self.grad(self.c[0]), self.grad(self.c[1])
        self.grho = self.grad(self.rho)
        lm = [self.lap(m) for m in self.mu]
        self.fa = (p["rho1"] - p["rho3"]) * self.mob[0] * lm[0] + (p["rho2"] - p["rho3"]) * self.mob[1] * lm[1]
        body = (p["gx"], p["gy"], 0.0)
        self.force = [(self.mu[0] - m3) * a + (self.mu[1] - m3) * b + self.rho * q for a, b, q in zip(g1, g2, body)]
        safe = torch.where(self.fluid, self.rho, 1.0)
        q = range(len(self.e))
        self.u = [(sum(self.e[k][b] * self.g[k] for k in q if self.e[k][b]) + 0.5 * self.force[b]) / safe
                  for b in range(self.d)]
        self.u = [torch.where(self.fluid, a, 0.0) for a in self.u]
        self.pr = (sum(self.g[1:]) + 0.5 * sum(a * b for a, b in zip(self.u, self.grho))
                   + self.rho * self.sk(0, self.u)) / (3 * (1 - self.w[0]))
        self.pr = torch.where(self.fluid, self.pr, 0.0)
        self.lower([self.pr, self.fa] + self.grho + self.force)
        if self.lid:
            self.u[0][-1] = torch.where(self.kind[-1] == TOP, p["lid_u"], self.u[0][-1])

    def relax(self, f, eq, src, rates):
        """BGK with one rate, or the moment basis of Lallemand and Luo with one rate per moment."""
        if not isinstance(rates, list):
            return [a - rates * (a - b) + (1 - rates / 2) * s for a, b, s in zip(f, eq, src)]
        rows = []
        for x, y in self.e:
            n = x * x + y * y
            rows.append([1, 3 * n - 4, (8 - 21 * n + 9 * n * n) / 2, x, (3 * n - 5) * x, y, (3 * n - 5) * y,
                         x * x - y * y, x * y])
        norm = (9, 36, 36, 6, 12, 6, 12, 4, 4)
        post = []
        for r in range(9):
            d = sum(rows[k][r] * (eq[k] - f[k]) for k in range(9) if rows[k][r])
            s = sum(rows[k][r] * src[k] for k in range(9) if rows[k][r])
            post.append((rates[r] * d + (1 - rates[r] / 2) * s) / norm[r])
        return [f[k] + sum(rows[k][r] * post[r] for r in range(9) if rows[k][r]) for k in range(9)]

    def step(self):
        self.macros()
        p, q, u, rho = self.p, range(len(self.e)), self.u, self.rho
        nu = self.c[0] * p["nu1"] + self.c[1] * p["nu2"] + (1 - self.c[0] - self.c[1]) * p["nu3"]
        rate = 1 / (3 * nu + 0.5)
        mrt = p["collision"] == 1.0
        cu = [[c * a for a in u] for c in self.c]
        f, g = self.f, self.g
        if self.lid:  # the lid row's populations from those of the row below
            f, g = [[a.clone() for a in fi] for fi in f], [a.clone() for a in g]
            top = self.kind[-1] == TOP
            above, under = [a[-1] for a in u], [a[-2] for a in u]
            for k in q:
                for i in range(2):
                    c, m = self.c[i][-2], self.mu[i][-2]
                    v = self.feq(i, k, c, m, above) + f[i][k][-2] - self.feq(i, k, c, m, under)
                    f[i][k][-1] = torch.where(top, v, f[i][k][-1])
                v = self.geq(k, self.pr[-2], rho[-2], above) + g[k][-2] - self.geq(k, self.pr[-2], rho[-2], under)
                g[k][-1] = torch.where(top, v, g[k][-1])
        post = []
        for i in range(2):
            d = [a - b for a, b in zip(cu[i], self.cu[i])]
            eq = [self.feq(i, k, self.c[i], self.mu[i], u) for k in q]
            src = [3 * self.w[k] * self.dot(k, d) for k in q]
            r = 1 / self.tau[i]
            post.append(self.relax(f[i], eq, src, [r if m in (0, 3, 5) else p["mrt_s_f"] for m in range(9)] if mrt else r))
        eq = [self.geq(k, self.pr, rho, u) for k in q]
        src = []
        for k in q:
            s = self.sk(k, u)
            src.append(sum((self.e[k][b] - u[b]) * (s * self.grho[b] + 3 * (s + self.w[k]) * self.force[b])
                           for b in range(self.d)))
        out = self.relax(g, eq, src, [p["mrt_s_g"] if m in (1, 2, 4, 6) else rate for m in range(9)] if mrt else rate)
        post.append([a + 3 * self.w[k] * self.fa * self.dot(k, u) for k, a in enumerate(out)])
        new = []
        for h in post:
            new.append([])
            for k in q:
                b = self.opp[k]
                v = torch.where(self.open[b], self.at(h[k], self.e[b]), torch.where(self.solid[b], h[b], 0.0))
                new[-1].append(torch.where(self.live, v, 0.0))
        self.f, self.g = new[:2], new[2]
        self.cu = cu

    def run(self, steps):
        for _ in range(steps):
            self.step()
        self.macros()
        return [torch.where(self.live, a, 0.0) for a in self.c + self.u + [self.pr]]
