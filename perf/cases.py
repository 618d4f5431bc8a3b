"""Timed cases of the lattice-Boltzmann library, through its public calls.

A pass is one solve as a program runs it: initial fields in device memory to
`lb_init`, `lb_step(n)`, the macroscopic fields with `lb_fields` (further
species with `lb_species_state`, cell types and liquid mass with
`lb_free_surface_state`) and the totals with `lb_reduce`. The batch family is
the serving loop's chunk instead: `lb_step_batch` of n steps over resident
lattices and the fields of each. What a program prepares once - the context,
with its porosity, permeability and solid cells, and where a case says `tune`
the timed choice of launch shape that the benchmark makes - is prepared here
too; everything else is in the pass. The number of steps is kept small against
a real run's thousands, so that a pass stays short; initialisation and export
are a few per cent of it.

Families (those of the repository's workloads):
  channel      FP64 Brinkman channel, walls, no solute
  wood         adhesive pressed into wood: full tensor K, pressure faces,
               solute inlet / outlet, hardening viscosity
  miscible     layered medium, diagonal K, solute inlet / outlet
  precision    the same with a full tensor K turned per 32^3 block
  forchheimer  coarse medium with inertial drag
  species      miscible with three solute species
  medium       every feature at once: impermeable cells, walls, full K, random
               initial velocity, optionally surface tension
  drop         free surface: liquid drop falling onto a wall
  batch        several miscible lattices of given sides stepped together

`exact` advances the same equations in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_0912_4230_gb300 import lb
from paper_0912_4230_gb300 import workloads as W

P, WALL, INLET, OUTLET, PRESSURE = W.PERIODIC, W.WALL, W.INLET, W.OUTLET, W.PRESSURE
PERIODIC3 = ((P, P), (P, P), (P, P))
LIQUID, INTERFACE, EMPTY = W.LIQUID, W.INTERFACE, W.EMPTY
Q = 19


def _c(name, family, nx, ny, nz, steps, storage="fp32", **kw):
    return dict(name=name, family=family, nx=nx, ny=ny, nz=nz, steps=steps, storage=storage, **kw)


def listed():
    return [
        # the smallest workload of the repository: launches and FP64 latency
        _c("channel_fp64", "channel", 16, 16, 64, 200, "fp64"),
        # the paper's own wood sample, one cell thick, odd rows
        _c("wood_sheet_fp64", "wood", 90, 90, 1, 120, "fp64", depth=60),
        # one small served request stepped alone
        _c("request_small", "miscible", 32, 32, 45, 300),
        # a serving chunk of small requests in 16-bit storage
        _c("serve_small_fp16", "batch", 0, 0, 0, 60, "fp16", sides="32x24"),
        # a serving chunk over mixed sizes (some fill the GPU alone)
        _c("serve_mix", "batch", 0, 0, 0, 30, "fp32", sides="32x6 48x4 64x3 96x1 128x1"),
        # the benchmark
        _c("miscible_128", "miscible", 128, 128, 128, 100, tune=True),
        # a user's own geometry: impermeable cells, walls, odd sizes
        _c("medium_ragged", "medium", 117, 83, 101, 60),
        # the largest: 16-bit storage of a full-tensor medium
        _c("precision_256_fp16", "precision", 256, 256, 256, 40, "fp16", tune=True),
        # three species sharing the flow
        _c("species_128", "species", 128, 128, 128, 60, tune=True),
        # inertial drag
        _c("forchheimer_128", "forchheimer", 128, 128, 128, 60, tune=True),
        # the wood sample at full size in FP32
        _c("wood_256", "wood", 256, 192, 64, 60, depth=128, tune=True),
        # free surface through the fall, the impact and the first spreading
        _c("drop_192", "drop", 192, 192, 128, 300, R=24.0, gap=3.0),
    ]


def draw(rng):
    """One more case of the same families and ranges."""
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def sides(cells):   # three sides of about that many cells, odd ones among them
        s = cells ** (1.0 / 3.0)
        nx = max(8, int(s * log(0.6, 1.6)))
        ny = max(5, int(s * log(0.7, 1.4)))
        return nx, ny, max(5, min(512, int(cells / (nx * ny))))

    def steps(cells, work):
        return int(min(100, max(8, work / cells)))

    fam = rng.choice(["channel", "wood", "miscible", "miscible", "precision", "precision",
                      "forchheimer", "species", "medium", "drop", "batch"])
    kw = {}
    if fam == "batch":
        total, parts = log(2e5, 4e6), []
        while total > 32768 and len(parts) < 4:
            side = rng.choice([s for s in (32, 40, 48, 64, 72, 96, 128) if s ** 3 <= total])
            k = rng.randint(1, max(1, min(12, int(total / side ** 3))))
            parts.append("%dx%d" % (side, k))
            total -= k * side ** 3
        return dict(family=fam, nx=0, ny=0, nz=0, steps=rng.randint(12, 40),
                    storage=rng.choice(["fp32", "fp16"]), sides=" ".join(parts))
    if fam == "drop":
        R = rng.uniform(8.0, 26.0)
        s = int(R * rng.uniform(4.5, 7.5))
        return dict(family=fam, nx=s + rng.randint(0, 17), ny=s, nz=int(4.2 * R),
                    steps=rng.randint(60, 300), storage=rng.choice(["fp32", "fp32", "fp64"]),
                    R=R, gap=rng.uniform(2.0, 6.0))
    if fam == "channel":
        storage = "fp64"
        nx, ny, nz = sides(log(6e3, 4e5))
    elif fam == "wood":
        storage = rng.choice(["fp64", "fp32"])
        nx, ny, nz = sides(log(8e3, 1.5e5 if storage == "fp64" else 4e6))
        ny = max(ny, 24)
        kw["depth"] = int(ny * 0.66)
    elif fam in ("miscible", "precision"):
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16", "fp64"])
        nx, ny, nz = sides(log(3e4, 1.5e5 if storage == "fp64" else 1.2e7))
    else:
        storage = "fp32"
        nx, ny, nz = sides(log(3e4, 4e6))
        if fam == "medium":
            storage = rng.choice(["fp32", "fp32", "fp16"])
            kw["A"] = rng.choice([0.0, 0.0, 1e-3])
    cells = nx * ny * nz
    work = 1e6 if storage == "fp64" else 6e7
    return dict(family=fam, nx=nx, ny=ny, nz=nz, steps=steps(cells, work), storage=storage,
                tune=rng.random() < 0.5 and not kw.get("A"), **kw)


# ------------------------------------------------------------------ inputs

def _cells(nx, ny, nz, dev):
    z = torch.arange(nz, device=dev).view(nz, 1, 1).expand(nz, ny, nx)
    y = torch.arange(ny, device=dev).view(1, ny, 1).expand(nz, ny, nx)
    x = torch.arange(nx, device=dev).view(1, 1, nx).expand(nz, ny, nx)
    return x, y, z


def _rotations(k, gen, dev):
    """Haar-random rotations from unit quaternions."""
    q = torch.randn(k, 4, generator=gen, device=dev, dtype=torch.float64)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)],
                       dim=1).view(k, 3, 3)


def _sym6(K):
    return torch.stack([K[..., 0, 0], K[..., 1, 1], K[..., 2, 2], K[..., 0, 1], K[..., 1, 2],
                        K[..., 2, 0]], dim=-1)


def _problem(case, seed, dev):
    """The workload of a case as a Problem whose arrays are tensors on dev."""
    fam, nx, ny, nz = case["family"], case["nx"], case["ny"], case["nz"]
    N, shape = nx * ny * nz, (nz, ny, nx)
    g = torch.Generator(device=dev).manual_seed(seed)

    def uni(lo, hi, *n):
        return torch.rand(*(n or shape), generator=g, device=dev) * (hi - lo) + lo

    x, y, z = _cells(nx, ny, nz, dev)
    bc = sbc = PERIODIC3
    K6 = C0 = cell_type = lambda0 = f_scale = None
    solid = torch.zeros(shape, dtype=torch.uint8, device=dev)
    rho0 = torch.ones(shape, device=dev)
    u0 = torch.zeros(shape + (3,), device=dev)
    if fam == "channel":
        bc = sbc = ((P, P), (P, P), (WALL, WALL))
        prm = dict(tau=0.8, G=(1e-6, 0.0, 0.0))
        eps = torch.full(shape, 0.6, device=dev)
        K6 = torch.zeros(shape + (6,), device=dev)
        K6[..., :3] = 1e-2
        u0[..., 0] = uni(0.0, 1e-8)
    elif fam == "wood":
        depth, dl = case["depth"], 30.0
        th = math.radians(45.0)
        r = (math.cos(th), math.sin(th))
        xi = torch.remainder((x * r[0] + y * r[1]).double() / dl, 1.0)
        rho_w = 310.0 * (1 + 1.24 * xi ** 0.2 * torch.exp(0.2 * xi)) * uni(0.99, 1.01)
        eps_w = 1 - rho_w / 1500.0
        f = (1500.0 / rho_w) ** 2 * eps_w ** (11.0 / 3.0) * 1e-3
        inw = (y < depth)
        kr, kl, kt = 8.2 * f, 51470.0 * f, 0.82 * f
        K6 = torch.stack([kr * r[0] ** 2 + kt * r[1] ** 2, kr * r[1] ** 2 + kt * r[0] ** 2, kl,
                          (kr - kt) * r[0] * r[1], 0 * kl, 0 * kl], dim=-1)
        iso = torch.tensor([1e6] * 3 + [0.0] * 3, device=dev, dtype=torch.float64)
        K6 = torch.where(inw[..., None], K6, iso).float()
        eps = torch.where(inw, eps_w, torch.ones_like(eps_w)).float()
        C0 = (~inw).float()
        P_top, P_bot = 1 / 3 + 0.0441, 1 / (3 * float(eps[:, 0, :].double().mean()))
        rho0 = torch.where(inw, 3 * eps * P_bot, torch.full_like(eps, 3 * P_top))
        bc, sbc = ((P, P), (PRESSURE, PRESSURE), (P, P)), ((P, P), (OUTLET, INLET), (P, P))
        prm = dict(visc_law=2, nu_g=0.15, a=2.05e-9, alpha=2e-3, beta=1e-3, solute=1, tau_D=0.8,
                   C_in=1.0, face_P=((0.0, 0.0), (P_bot, P_top), (0.0, 0.0)))
    elif fam == "drop":
        R, gap = case["R"], case["gap"]
        c = ((nx - 1) / 2, (ny - 1) / 2, 0.5 + gap + R)
        solid[0] = 1
        lq = ((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2 <= R * R) & (solid == 0)
        near = torch.zeros_like(lq)
        for q in range(1, Q):
            near |= torch.roll(lq, (CZ[q], CY[q], CX[q]), (0, 1, 2))
        near[0] = near[-1] = False
        cell_type = torch.full(shape, EMPTY, dtype=torch.uint8, device=dev)
        cell_type[near] = INTERFACE
        cell_type[lq] = LIQUID
        lambda0 = torch.where(lq, 1.0, torch.where(near, 0.5, 0.0)).float()
        u0[..., 2] = -0.02 * (cell_type != EMPTY)
        bc = sbc = ((P, P), (P, P), (WALL, WALL))
        prm = dict(tau=0.7, A=1e-3, wall_rho=0.6, free_surface=1)
        eps = torch.ones(shape, device=dev)
        f_scale = 1 + 0.01 * uni(-1.0, 1.0, Q, *shape)
    else:
        # the layered medium: porosity bands of period 16 along x with noise,
        # K log-uniform per cell and 100 (coarse: 10) times larger along z
        eps = torch.where((x % 16) < 8, 0.35, 0.85) + uni(-0.05, 0.05)
        k = 10 ** (uni(-2.0, 0.0) if fam == "forchheimer" else uni(-4.0, -2.0))
        K6 = torch.zeros(shape + (6,), device=dev)
        K6[..., 0] = K6[..., 1] = k
        K6[..., 2] = (10 if fam == "forchheimer" else 100) * k
        C0 = torch.zeros(shape, device=dev)
        sbc = ((P, P), (P, P), (INLET, OUTLET))
        prm = dict(visc_law=1, tau0=0.6, tau1=1.5, G=(0.0, 0.0, 1e-5), solute=1, tau_D=0.8,
                   C_in=1.0)
        if fam == "forchheimer":
            prm.update(G=(0.0, 0.0, 1e-4), forchheimer=1.0)
        if fam == "species":
            prm.update(species=3, species_tau_D=(0.0, 1.2, 0.6), species_C_in=(0.0, 0.5, 0.0))
            C0 = torch.stack([C0, C0, torch.full(shape, 0.3, device=dev)])
        if fam in ("precision", "medium"):
            nb = [-(-n // 32) for n in (nx, ny, nz)]
            Rb = _rotations(nb[0] * nb[1] * nb[2], g, dev).float()
            b = ((x // 32) + nb[0] * ((y // 32) + nb[1] * (z // 32))).reshape(-1)
            t = _sym6(torch.einsum("bi,bj->bij", Rb[:, :, 2], Rb[:, :, 2]))
            one = torch.tensor([1.0] * 3 + [0.0] * 3, device=dev)
            K6 = (k.reshape(-1, 1) * (99 * t[b] + one)).view(shape + (6,))
        if fam == "medium":
            eps = uni(0.3, 1.0)
            solid = (uni(0.0, 1.0) < 0.1).to(torch.uint8)
            bc, sbc = ((P, P), (WALL, WALL), (P, P)), ((P, P), (WALL, WALL), (INLET, OUTLET))
            rho0, u0 = uni(0.99, 1.01), uni(-0.02, 0.02, *shape, 3)
            C0 = uni(0.0, 1.0)
            prm.update(tau0=0.7, tau1=1.3, G=(2e-4, -1e-4, 3e-4), tau_D=0.75,
                       A=case.get("A", 0.0), wall_rho=0.3)
    return W.Problem(name=fam, nx=nx, ny=ny, nz=nz, bc=bc, sbc=sbc, params=prm,
                     eps=eps.contiguous(), K6=None if K6 is None else K6.contiguous(),
                     solid=solid, rho0=rho0.contiguous(), u0=u0.contiguous(), C0=C0,
                     cell_type=cell_type, lambda0=lambda0, f_scale=f_scale,
                     storage=case["storage"])


def _members(case):
    """The lattices of a batch case, as cases of their own."""
    out = []
    for part in case["sides"].split():
        side, k = (int(v) for v in part.split("x"))
        # served domains are cubes stretched along z (aspect 1 to 2)
        out += [dict(case, family="miscible", nx=side, ny=side, nz=side + (5 * side) // 16 * (i % 2))
                for i in range(k)]
    return out


class Solve:
    """A context and the arrays a program keeps beside it."""

    def __init__(self, case, seed):
        p = self.prob = _problem(case, seed, "cuda")
        self.case, self.ctx = case, None
        self.ctx = lb.lb_create(lb.make_domain(p), p.eps, p.K6, p.solid,
                                lb.make_params(p, check_every=1))
        N = p.N
        self.species = int(p.params.get("species", 1))
        self.rho, self.C, self.nu = (torch.zeros(N, device="cuda") for _ in range(3))
        self.u = torch.zeros(3 * N, device="cuda")
        self.Cs = [torch.zeros(N, device="cuda") for _ in range(self.species - 1)]
        if p.cell_type is not None:
            self.type = torch.zeros(N, dtype=torch.uint8, device="cuda")
            self.mass = torch.zeros(N, dtype=torch.float64, device="cuda")
        self.init()
        if case.get("tune"):
            lb.lb_autotune(self.ctx, 3)

    def init(self):
        p = self.prob
        lb.lb_init(self.ctx, p.rho0, p.u0, p.C0, p.cell_type, p.lambda0, p.f_scale)

    def fields(self):
        lb.lb_fields(self.ctx, self.rho, self.u, self.C, self.nu)
        return {"rho": self.rho, "u": self.u, "C": self.C, "nu": self.nu}

    def __del__(self):
        if self.ctx is not None:
            lb.lb_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    if case["family"] == "batch":
        return [Solve(c, seed * 1000 + i) for i, c in enumerate(_members(case))]
    return Solve(case, seed)


def run(state):
    if isinstance(state, list):
        lb.lb_step_batch([s.ctx for s in state], state[0].case["steps"])
        out = [s.fields() for s in state]
        # the fields of all lattices, member after member
        return {k: torch.cat([o[k] for o in out]) for k in ("rho", "u", "C", "nu")}
    s = state
    s.init()
    lb.lb_step(s.ctx, s.case["steps"])
    out = s.fields()
    # totals of 32- and 16-bit populations carry 32 bits
    exact64 = s.case["storage"] == "fp64"
    out["totals"] = lb.lb_reduce(s.ctx).astype(np.float64 if exact64 else np.float32)
    for k, C in enumerate(s.Cs):
        lb.lb_species_state(s.ctx, k + 1, C)
        out["C%d" % (k + 1)] = C
    if s.prob.cell_type is not None:
        lb.lb_free_surface_state(s.ctx, s.type, s.mass)
        out["type"], out["mass"] = s.type, s.mass if exact64 else s.mass.float()
    return out


def work(case):
    """Every step reads and writes each population of every updated cell once
    and reads its static fields once (a state larger than the chip's memory
    has to); the pass also reads the initial fields, writes the first state
    and writes the exported fields."""
    if case["family"] == "batch":
        ws = [work(c) for c in _members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    fam, steps = case["family"], case["steps"]
    N = case["nx"] * case["ny"] * case["nz"]
    e = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case["storage"]]
    real = 8 if e == 8 else 4
    if fam == "drop":
        R = case["R"]
        live = 4.19 * R ** 3 + 12.6 * R * R * 1.5   # liquid and interface cells
        return {"bytes": steps * live * (2 * Q * e + 4 * real + 3) + N * 29,
                "flops": steps * live * 420}
    lattices = {"channel": 1, "species": 4}.get(fam, 2)
    rows = 6 if fam in ("precision", "wood", "medium") else 3
    pops = lattices * Q * e
    step = 2 * pops + (1 + rows) * real + 1
    flops = 260 + 110 * (lattices - 1) + (60 if rows == 6 else 20) + (140 if fam == "forchheimer" else 0)
    once = 4 * (4 + max(0, lattices - 1)) + pops + 4 * (5 + max(1, lattices - 1))
    return {"bytes": N * (steps * step + once), "flops": N * steps * flops}


# ------------------------------------------------- the same in 64 bits (torch)

def _directions():
    c = [(0, 0, 0)]
    for a, b in ((0, 1), (1, 2), (2, 0)):
        for s, t in ((1, 1), (-1, 1), (-1, -1), (1, -1), (1, 0), (-1, 0)):
            v = [0, 0, 0]
            v[a], v[b] = s, t
            c.append(tuple(v))
    return c


DIRS = _directions()
CX, CY, CZ = ([d[i] for d in DIRS] for i in range(3))
OPP = [DIRS.index(tuple(-v for v in d)) for d in DIRS]
WT = [{0: 1 / 3, 1: 1 / 18, 2: 1 / 36}[sum(abs(v) for v in d)] for d in DIRS]


def _behind(a, q):
    """a at x - c_q (wrapped)."""
    return torch.roll(a, (CZ[q], CY[q], CX[q]), (-3, -2, -1))


def _ahead(a, q):
    return torch.roll(a, (-CZ[q], -CY[q], -CX[q]), (-3, -2, -1))


def _dot(q, v):
    s = 0.0
    for d, a in zip(DIRS[q], v):
        if d:
            s = s + d * a
    return s


def _masks(p, kinds, wanted):
    """Per direction: cells whose pull x - c_q leaves the box through a face of a kind in `wanted`."""
    x, y, z = _cells(p.nx, p.ny, p.nz, p.eps.device)
    out = []
    for d in DIRS:
        m = None
        for v, c, n, faces in ((d[0], x, p.nx, kinds[0]), (d[1], y, p.ny, kinds[1]), (d[2], z, p.nz, kinds[2])):
            if v and faces[0 if v > 0 else 1] in wanted:
                e = c == (0 if v > 0 else n - 1)
                m = e if m is None else m | e
        out.append(m)
    return out


def _or(*ms):
    r = None
    for m in ms:
        if m is not None:
            r = m if r is None else r | m
    return r


def _feq(q, rho, V, ie, uu, st=None):
    cu = _dot(q, V)
    e = WT[q] * rho * (1 + 3 * cu + 4.5 * ie * cu * cu - 1.5 * ie * uu)
    if st is not None:   # surface tension: (A eps tau, F, |F|, its inverse or 0)
        stc, F, Fn, iF = st
        e = e + (WT[0] * stc * Fn if q == 0 else WT[q] * stc * (_dot(q, F) ** 2 * iF - Fn))
    return e


def _gradient(field, wall_rho, walls):
    """sum_q field(x + c_q) c_q; a step out through a wall sees wall_rho."""
    F = [torch.zeros_like(field) for _ in range(3)]
    for q in range(1, Q):
        r = _ahead(field, q)
        if walls[OPP[q]] is not None:
            r = torch.where(walls[OPP[q]], torch.full_like(r, wall_rho), r)
        for i in range(3):
            if DIRS[q][i]:
                F[i] += DIRS[q][i] * r
    return F


def _tension(A, eps, tau, F):
    Fn = (F[0] ** 2 + F[1] ** 2 + F[2] ** 2).sqrt()
    on = Fn > 1e-20
    return torch.where(on, A * eps * tau, 0.0), F, Fn, torch.where(on, 1 / Fn.clamp_min(1e-30), 0.0)


def _collide_fluid(fs, rho, V, Fe, ie, tau, st):
    uu = V[0] ** 2 + V[1] ** 2 + V[2] ** 2
    uF = V[0] * Fe[0] + V[1] * Fe[1] + V[2] * Fe[2]
    for q in range(Q):
        cu, cF = _dot(q, V), _dot(q, Fe)
        T = WT[q] * rho * (1 - 0.5 / tau) * (3 * cF + 9 * ie * cu * cF - 3 * ie * uF)
        fs[q] = fs[q] - (fs[q] - _feq(q, rho, V, ie, uu, st)) / tau + T


def _inverse6(K):
    a, b, c, d, e, f = (v.double() for v in K.unbind(-1))   # xx yy zz xy yz zx
    m = [b * c - e * e, a * c - f * f, a * b - d * d, f * e - d * c, d * f - a * e, d * e - b * f]
    det = a * m[0] + d * m[3] + f * m[5]
    return [v / det for v in m]


def _velocity(k, eps, nu, V, G, cF):
    r = [V[i] + 0.5 * eps * G[i] for i in range(3)]
    if cF:
        # V'_i = r_i / (a_i + b_i s) with s = |V'|: Newton from below, where
        # s - |V'(s)| is concave and increasing
        Fe = cF * 1.75 / (150 * eps ** 3).sqrt()
        a = [1 + 0.5 * eps * nu * k[i] for i in range(3)]
        b = [0.5 * eps * Fe * k[i].sqrt() for i in range(3)]
        s = torch.zeros_like(eps)
        for _ in range(10):
            v = [r[i] / (a[i] + b[i] * s) for i in range(3)]
            n = (v[0] ** 2 + v[1] ** 2 + v[2] ** 2).sqrt().clamp_min(1e-300)
            g = sum(v[i] ** 2 * b[i] / (a[i] + b[i] * s) for i in range(3))
            s = s - (s - n) / (1 + g / n)
        Vp = [r[i] / (a[i] + b[i] * s) for i in range(3)]
    else:
        h = 0.5 * eps * nu
        L = [1 + h * k[0], 1 + h * k[1], 1 + h * k[2], h * k[3], h * k[4], h * k[5]]
        m = [L[1] * L[2] - L[4] ** 2, L[0] * L[2] - L[5] ** 2, L[0] * L[1] - L[3] ** 2,
             L[5] * L[4] - L[3] * L[2], L[3] * L[5] - L[0] * L[4], L[3] * L[4] - L[1] * L[5]]
        det = L[0] * m[0] + L[3] * m[3] + L[5] * m[5]
        Vp = [(m[0] * r[0] + m[3] * r[1] + m[5] * r[2]) / det,
              (m[3] * r[0] + m[1] * r[1] + m[4] * r[2]) / det,
              (m[5] * r[0] + m[4] * r[1] + m[2] * r[2]) / det]
    # V' = V + F^ext / 2
    return Vp, [2 * (Vp[i] - V[i]) for i in range(3)]


def _porous64(p, steps):
    """All families but the drop."""
    prm, dev = p.params, p.eps.device
    solid = p.solid.bool()
    eps = torch.where(solid, 1.0, p.eps.double())
    ie, k, G = 1 / eps, _inverse6(p.K6), prm["G"] if "G" in prm else (0.0,) * 3
    k = [torch.where(solid, 1.0 if i < 3 else 0.0, v) for i, v in enumerate(k)]
    law, sol, A = prm.get("visc_law", 0), prm.get("solute", 0), prm.get("A", 0.0)
    S = int(prm.get("species", 1)) if sol else 0
    tD = [prm.get("tau_D", 1.0)] + list(prm.get("species_tau_D", ()))[1:]
    Cin = [prm.get("C_in", 0.0)] + list(prm.get("species_C_in", ()))[1:]
    any_solid = bool(solid.any())
    sol_src = [_behind(solid, q) if any_solid and q else None for q in range(Q)]
    f_wall, f_press = _masks(p, p.bc, (WALL,)), _masks(p, p.bc, (PRESSURE,))
    s_wall, s_in, s_out = (_masks(p, p.sbc, (v,)) for v in (WALL, INLET, OUTLET))
    closed = _masks(p, p.sbc, (WALL, INLET, OUTLET))
    ge = []
    if sol:   # grad(eps)/eps with the cell's own porosity at solid or outside neighbours
        ge = [torch.zeros_like(eps) for _ in range(3)]
        for q in range(1, Q):
            e = _ahead(eps, q)
            m = _or(closed[OPP[q]], sol_src[OPP[q]])
            if m is not None:
                e = torch.where(m, eps, e)
            for i in range(3):
                if DIRS[q][i]:
                    ge[i] += 3 * WT[q] * DIRS[q][i] * e
        ge = [v * ie for v in ge]

    def tau_of(C, t):
        if law == 1:
            return prm["tau0"] + (prm["tau1"] - prm["tau0"]) * C.clamp(0.0, 1.0)
        if law == 2:
            nu = prm["nu_g"] * (1 + prm["a"] * math.exp(prm["alpha"] * t)) * torch.exp(prm["beta"] * (1 - C))
            return 3 * nu + 0.5
        return torch.full_like(eps, prm["tau"])

    u0 = [v.double() for v in p.u0.unbind(-1)]
    rho0 = p.rho0.double()
    C0 = [] if not sol else [v.double() for v in (p.C0 if S > 1 else p.C0[None])]
    st = None
    if A:
        st = _tension(A, eps, tau_of(C0[0], 0), _gradient(torch.where(solid, prm["wall_rho"], rho0), prm["wall_rho"], f_wall))
    uu = u0[0] ** 2 + u0[1] ** 2 + u0[2] ** 2
    f = [torch.where(solid, 0.0, _feq(q, rho0, u0, ie, uu, st)) for q in range(Q)]
    h = []
    for s in range(S):
        D = (tD[s] - 0.5) / 3
        v = [u0[i] + D * ge[i] for i in range(3)]
        h.append([torch.where(solid, 0.0, WT[q] * eps * C0[s] * (1 + 3 * _dot(q, v))) for q in range(Q)])
    flux = [0.0, 0.0]
    for t in range(1, steps + 1):
        own = None
        if any(m is not None for m in f_press):
            r = sum(f)
            own = r, [sum(DIRS[q][i] * f[q] for q in range(Q) if DIRS[q][i]) / r for i in range(3)]
        fs = []
        for q in range(Q):
            v, m = _behind(f[q], q), _or(f_wall[q], sol_src[q])
            if m is not None:
                v = torch.where(m, f[OPP[q]], v)
            if f_press[q] is not None:   # one axis only in these cases
                u = own[1]
                a = [i for i in range(3) if DIRS[q][i] and p.bc[i][0] == PRESSURE][0]
                rb = 3 * eps * prm["face_P"][a][0 if DIRS[q][a] > 0 else 1]
                cu, w2 = _dot(q, u), u[0] ** 2 + u[1] ** 2 + u[2] ** 2
                e = 2 * WT[q] * rb * (1 + 4.5 * ie * cu * cu - 1.5 * ie * w2)
                v = torch.where(f_press[q], e - f[OPP[q]], v)
            fs.append(v)
        rho = torch.where(solid, 1.0, sum(fs))
        V = [sum(DIRS[q][i] * fs[q] for q in range(Q) if DIRS[q][i]) / rho for i in range(3)]
        hs, sC = [], []
        for s in range(S):
            D = (tD[s] - 0.5) / 3
            vi = [V[i] + D * ge[i] for i in range(3)]
            new = []
            for q in range(Q):
                v, b = _behind(h[s][q], q), h[s][OPP[q]]
                if sol_src[q] is not None:
                    v = torch.where(sol_src[q], b, v)
                if s_out[q] is not None:
                    v = torch.where(s_out[q], h[s][q], v)
                if s_in[q] is not None:
                    v = torch.where(s_in[q], WT[q] * eps * Cin[s] * (1 + 3 * _dot(q, vi)), v)
                if s_wall[q] is not None:
                    v = torch.where(s_wall[q], b, v)
                if s == 0:
                    for i, (m, sg) in enumerate(((s_in[q], 1.0), (s_out[q], -1.0))):
                        if m is not None:
                            m = m & ~solid
                            if i == 1 and s_in[q] is not None:
                                m = m & ~s_in[q]
                            if s_wall[q] is not None:
                                m = m & ~s_wall[q]
                            flux[i] += float((sg * (v - b))[m].sum())
                new.append(v)
            hs.append(new)
            sC.append(sum(new))
        C = sC[0] * ie if sol else torch.zeros_like(eps)
        tau = tau_of(C, t)
        nu = (tau - 0.5) / 3
        st = None
        if A:
            st = _tension(A, eps, tau, _gradient(torch.where(solid, prm["wall_rho"], rho), prm["wall_rho"], f_wall))
        Vp, Fe = _velocity(k, eps, nu, V, G, prm.get("forchheimer", 0.0))
        _collide_fluid(fs, rho, Vp, Fe, ie, tau, st)
        f = fs
        for s in range(S):
            D = (tD[s] - 0.5) / 3
            v = [Vp[i] + D * ge[i] for i in range(3)]
            for q in range(Q):
                hs[s][q] = hs[s][q] - (hs[s][q] - WT[q] * sC[s] * (1 + 3 * _dot(q, v))) / tD[s]
        h = hs

    def live(v):
        return torch.where(solid, 0.0, v).reshape(-1)

    out = {"rho": live(rho), "u": torch.where(solid[..., None], 0.0, torch.stack(Vp, -1)).reshape(-1),
           "C": live(C), "nu": live(nu)}
    mass = float(sum(v[~solid].sum() for v in f))
    solute = float(sum(v[~solid].sum() for v in h[0])) if sol else 0.0
    out["totals"] = np.array([mass, solute] + flux)
    for s in range(1, S):
        out["C%d" % s] = live(sC[s] * ie)
    return out


def _drop64(p, steps):
    """Free surface: eps = 1, no body force, walls along z, one solid layer."""
    prm = p.params
    tau, A, wall_rho = prm["tau"], prm["A"], prm["wall_rho"]
    solid = p.solid.bool()
    walls = _masks(p, p.bc, (WALL,))
    # per direction: the neighbour x + c_q exists and is not solid; the source x - c_q likewise
    shut = [_or(walls[q], _behind(solid, q)) for q in range(Q)]
    one = torch.ones_like(p.eps, dtype=torch.float64)
    typ = torch.where(solid, torch.full_like(p.cell_type, EMPTY), p.cell_type)
    lam = torch.where(typ == LIQUID, 1.0, torch.where(typ == INTERFACE, p.lambda0.double(), 0.0))
    m = lam * p.rho0.double()
    u0 = [v.double() for v in p.u0.unbind(-1)]
    uu = u0[0] ** 2 + u0[1] ** 2 + u0[2] ** 2
    st = _tension(A, one, tau, _gradient(torch.where(solid, wall_rho, m), wall_rho, walls))
    dead = typ == EMPTY
    f = [torch.where(dead, 0.0, _feq(q, p.rho0.double(), u0, 1.0, uu, st) * p.f_scale.view((Q,) + typ.shape)[q])
         for q in range(Q)]
    rho, Vp = torch.where(dead, 0.0, p.rho0.double()), [torch.where(dead, 0.0, v) for v in u0]
    for _ in range(steps):
        dead = typ == EMPTY
        own = torch.where(dead, 1.0, sum(f))
        u = [sum(DIRS[q][i] * f[q] for q in range(Q) if DIRS[q][i]) / own for i in range(3)]
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        dm, fs = torch.zeros_like(m), [f[0]]
        face = typ == INTERFACE
        for q in range(1, Q):
            o, ty = OPP[q], _ahead(typ, q)
            w = torch.where(face & (ty == INTERFACE), 0.5 * (lam + _ahead(lam, q)), 1.0)
            dm += torch.where(shut[o] | (ty == EMPTY), 0.0, w * (_ahead(f[o], q) - f[q]))
            gas = _feq(q, 1.0, u, 1.0, uu) + _feq(o, 1.0, u, 1.0, uu) - f[o]
            v = torch.where(_behind(dead, q), gas, _behind(f[q], q))
            fs.append(torch.where(shut[q], f[o], v))
        m = torch.where(dead, m, m + dm)
        r = torch.where(dead, 1.0, sum(fs))
        V = [torch.where(dead, 0.0, sum(DIRS[q][i] * fs[q] for q in range(Q) if DIRS[q][i]) / r) for i in range(3)]
        field = torch.where(solid, wall_rho, torch.where(dead, 0.0, m))
        st = _tension(A, one, tau, _gradient(field, wall_rho, walls))
        zero = [torch.zeros_like(m)] * 3
        _collide_fluid(fs, r, V, zero, 1.0, tau, st)
        f = [torch.where(dead, a, b) for a, b in zip(f, fs)]
        rho = torch.where(dead, rho, r)
        Vp = [torch.where(dead, a, b) for a, b in zip(Vp, V)]
        lam = torch.where(face, m / r, lam)
        fill, drain = face & (lam > 1.001), face & (lam < -0.001)

        def beside(flag):   # some neighbour x + c_q is flagged
            hit = torch.zeros_like(flag)
            for q in range(1, Q):
                hit |= _ahead(flag, q) & ~shut[OPP[q]]
            return hit

        if bool((fill | drain).any()):
            by_fill = beside(fill)
            drain &= ~by_fill
            new = dead & ~solid & by_fill
            back = (typ == LIQUID) & beside(drain)
            typ = torch.where(fill, torch.full_like(typ, LIQUID),
                              torch.where(drain, torch.full_like(typ, EMPTY),
                                          torch.where(new | back, torch.full_like(typ, INTERFACE), typ)))
            okay = (typ != EMPTY) & ~new & ~solid
            cnt, acc = torch.zeros_like(m), [torch.zeros_like(m) for _ in range(4)]
            nif = torch.zeros_like(m)
            for q in range(1, Q):
                a = (_ahead(okay, q) & ~shut[OPP[q]]).double()
                cnt += a
                for i, v in enumerate([rho] + Vp):
                    acc[i] += a * _ahead(v, q)
                nif += (_ahead(typ == INTERFACE, q) & ~shut[OPP[q]]).double()
            ic = 1 / cnt.clamp_min(1.0)
            nr, nu = torch.where(cnt > 0, acc[0] * ic, 1.0), [v * ic for v in acc[1:]]
            nn = nu[0] ** 2 + nu[1] ** 2 + nu[2] ** 2
            f = [torch.where(new, _feq(q, nr, nu, 1.0, nn), f[q]) for q in range(Q)]
            rho = torch.where(new, nr, rho)
            Vp = [torch.where(new, a, b) for a, b in zip(nu, Vp)]
            gone = (fill | drain) & (nif > 0)
            excess = torch.where(gone, torch.where(fill, m - rho, m), 0.0)
            m = m - excess
            share = excess / nif.clamp_min(1.0)
            got = torch.zeros_like(m)
            for q in range(1, Q):
                got += torch.where(shut[OPP[q]], 0.0, _ahead(share, q))
            m = torch.where((typ == INTERFACE) & ~solid, m + got, m)
            gone = typ == EMPTY
            rho = torch.where(gone, 0.0, rho)
            Vp = [torch.where(gone, 0.0, v) for v in Vp]
        lam = torch.where(typ == LIQUID, 1.0, torch.where(typ == EMPTY, 0.0, m / rho.clamp_min(1e-30)))
    nu = torch.where(typ == EMPTY, 0.0, (tau - 0.5) / 3)
    return {"rho": rho.reshape(-1), "u": torch.stack(Vp, -1).reshape(-1), "C": torch.zeros_like(rho).reshape(-1),
            "nu": nu.reshape(-1), "totals": np.array([float(m[~solid].sum()), 0.0, 0.0, 0.0]),
            "type": typ.reshape(-1), "mass": m.reshape(-1)}


def exact(case, seed):
    if case["family"] == "batch":
        out = [_porous64(_problem(c, seed * 1000 + i, "cuda"), case["steps"])
               for i, c in enumerate(_members(case))]
        return {k: torch.cat([o[k] for o in out]) for k in ("rho", "u", "C", "nu")}
    p = _problem(case, seed, "cuda")
    return _drop64(p, case["steps"]) if case["family"] == "drop" else _porous64(p, case["steps"])
