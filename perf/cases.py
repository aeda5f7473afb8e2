"""The work that users of this framework have it do, as timed cases.

A pass is what a simulation does between two looks at its flow: `steps` time steps of a Solver,
the FP64 sums of the final state, and the moments of the whole lattice read back on the GPU. With
"restart" the pass also loads the initial state first, as an ensemble of short runs does. The
adjoint cases are one gradient evaluation of an optimisation: forward rollout, loss, backward.

exact() is the same flow in plain 64-bit torch: populations rebuilt, streamed and projected one
direction at a time, and autograd (with recomputed segments) for the gradients.
"""
import math

import torch
import torch.utils.checkpoint

from paper_2609_09160_gb300 import Solver, rollout

DEV = "cuda"
SYM = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
STORED = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}


def _case(name, kind, lattice, storage, nx, ny, nz, tau, steps, **more):
    return dict(name=name, kind=kind, lattice=lattice, storage=storage, nx=nx, ny=ny, nz=nz, tau=tau, steps=steps, **more)


def listed():
    return [
        # validation run: the FP64 Taylor-Green decay, many short steps from a fresh state
        _case("tg32_d3q19_f64", "periodic", "19", "f64", 32, 32, 32, 0.8, 100, restart=True),
        # ensemble member: a small walled duct, where a step is a few microseconds
        _case("channel64_d3q19_f32", "channel", "19", "f32", 64, 48, 40, 0.9, 100, restart=True),
        # the headline production run: walled channel driven by a body force
        _case("channel256_d3q19_f32", "channel", "19", "f32", 256, 256, 256, 0.9, 20, restart=False),
        # walled channel of uneven size with 16-bit stored moments
        _case("channel_uneven_d3q19_bf16", "channel", "19", "bf16", 200, 163, 187, 0.8, 20, restart=False),
        # periodic box of odd size: rows that start on no 16-byte boundary
        _case("box_odd_d3q19_f32", "periodic", "19", "f32", 333, 250, 189, 0.6, 20, restart=False),
        # the largest runs: periodic turbulence-like flow, FP32 and FP16 stored
        _case("tg512_d3q27_f32", "periodic", "27", "f32", 512, 512, 512, 0.55, 20, restart=False),
        _case("tg512_d3q27_f16", "periodic", "27", "f16", 512, 512, 512, 0.55, 20, restart=False),
        # the complete Hermite basis (Galilean-invariant viscosity)
        _case("tg256_d3q27h_f32", "periodic", "27h", "f32", 256, 256, 256, 0.55, 20, restart=False),
        # flow through a porous medium: solid sites scattered over the whole lattice
        _case("porous_d3q19_f32", "porous", "19", "f32", 192, 160, 176, 0.8, 20, restart=False, solid=0.2),
        # two components at equal densities: a static droplet
        _case("droplet128_d3q19_f32", "droplet", "19", "f32", 128, 128, 128, 1.0, 50, restart=False),
        # two components with density and viscosity contrast between walls
        _case("layered_d3q19_f32", "layered", "19", "f32", 512, 1024, 8, 0.65, 50, restart=False),
        # gradient of a flow objective with respect to a force field and the initial state
        _case("adjoint128_d3q19_f32", "adjoint", "19", "f32", 128, 64, 64, 0.9, 500, every=50),
    ]


def _sizes(rng, sites):
    """Three extents whose product is about `sites`, none dominating; odd ones as often as even ones."""
    side = sites ** (1.0 / 3.0)
    a, b = 2.0 ** rng.uniform(-0.6, 0.6), 2.0 ** rng.uniform(-0.6, 0.6)
    nx, ny, nz = side * a, side * b, side / (a * b)
    return [max(8, int(round(v)) + rng.randrange(0, 2)) for v in (nx, ny, nz)]


def draw(rng):
    kind = rng.choice(("periodic", "periodic", "periodic", "channel", "channel", "porous", "droplet", "layered", "adjoint"))
    lattice = {"periodic": rng.choice(("19", "27", "27h")), "channel": rng.choice(("19", "27"))}.get(kind, "19")
    storage = rng.choice(("f64", "f32", "f32", "f16", "bf16")) if kind in ("periodic", "channel") else "f32"
    top = 18 if storage == "f64" else {"periodic": 25, "channel": 25, "porous": 23, "droplet": 22, "layered": 22, "adjoint": 19}[kind]
    nx, ny, nz = _sizes(rng, 2.0 ** rng.uniform(15, top))
    if rng.random() < 0.5:  # rows of whole 16-byte units, as most users choose them
        nx = (nx + 7) // 8 * 8
    steps = max(10, min(100, int(2 ** 28 / (nx * ny * nz))))
    c = dict(kind=kind, lattice=lattice, storage=storage, nx=nx, ny=ny, nz=nz, tau=round(rng.uniform(0.56, 1.1), 3), steps=steps)
    if kind == "adjoint":
        c["every"] = rng.randrange(10, 51)
        c["steps"] = rng.randrange(20, 201)
    else:
        c["restart"] = rng.random() < 0.3
    if kind == "porous":
        c["solid"] = round(rng.uniform(0.05, 0.35), 3)
    return c


# --------------------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _grid(shape):
    nz, ny, nx = shape
    ax = [torch.arange(n, dtype=torch.float32, device=DEV) for n in (nx, ny, nz)]
    return ax[0].reshape(1, 1, nx), ax[1].reshape(1, ny, 1), ax[2].reshape(nz, 1, 1)


def _vortices(shape, tau, seed):
    """Taylor-Green vortex (U0 = 0.04) plus eight solenoidal waves of random phase (0.01 in all):
    p*, u and the second moments u u - (tau / 3) (grad u + grad u^T) of a developed flow."""
    nz, ny, nx = shape
    x, y, z = (c * (2 * math.pi / n) for c, n in zip(_grid(shape), (nx, ny, nz)))
    h = (2 * math.pi / nx, 2 * math.pi / ny, 2 * math.pi / nz)
    M = torch.zeros((10,) + shape, device=DEV)
    sx, cx, sy, cy, cz, sz = x.sin(), x.cos(), y.sin(), y.cos(), z.cos(), z.sin()
    u0 = 0.04
    M[0] = 3 * u0 * u0 / 16 * ((2 * x).cos() + (2 * y).cos()) * (2 + (2 * z).cos())
    M[1] = u0 * sx * cy * cz
    M[2] = -u0 * cx * sy * cz
    g = -tau / 3.0
    M[4] = g * 2 * u0 * h[0] * (cx * cy * cz)
    M[5] = -g * 2 * u0 * h[1] * (cx * cy * cz)
    M[7] = g * u0 * (h[0] - h[1]) * (sx * sy * cz)
    M[8] = -g * u0 * h[2] * (sx * cy * sz)
    M[9] = g * u0 * h[2] * (cx * sy * sz)
    r = torch.Generator().manual_seed(int(seed))
    for _ in range(8):
        k = torch.randint(1, 5, (3,), generator=r) * (torch.randint(0, 2, (3,), generator=r) * 2 - 1)
        kv = torch.tensor([float(k[a]) * h[a] for a in range(3)])
        d = torch.linalg.cross(kv, torch.randn(3, generator=r))
        d = (d / d.norm() * 0.005).tolist()
        t = float(k[0]) * x + float(k[1]) * y + float(k[2]) * z + float(torch.rand((), generator=r)) * 2 * math.pi
        s, c = t.sin(), t.cos()
        kv = kv.tolist()
        for a in range(3):
            M[1 + a].add_(s, alpha=d[a])
        for i, (a, b) in enumerate(SYM):
            M[4 + i].add_(c, alpha=g * (d[a] * kv[b] + d[b] * kv[a]))
        del t, s, c
    for i, (a, b) in enumerate(SYM):
        M[4 + i].addcmul_(M[1 + a], M[1 + b])
    return M


def _noise(shape, seed):
    M = torch.zeros((10,) + shape, device=DEV)
    M[0].uniform_(-1e-3, 1e-3, generator=_gen(seed))
    return M


def _inputs(case, seed):
    """Initial moments, host mask, phase field, two-component parameters and uniform force."""
    shape = (case["nz"], case["ny"], case["nx"])
    nz, ny, nx = shape
    mask = phi = two = None
    force = (0.0, 0.0, 0.0)
    r = torch.Generator().manual_seed(int(seed) + 7)
    if case["kind"] == "periodic":
        M = _vortices(shape, case["tau"], seed)
    else:
        M = _noise(shape, seed)
    if case["kind"] in ("channel", "adjoint"):
        mask = torch.zeros(shape, dtype=torch.bool)
        mask[:, 0] = mask[:, -1] = True
        force = (1e-6, 0.0, 0.0) if case["kind"] == "channel" else force
    elif case["kind"] == "porous":
        mask = (torch.rand(shape, device=DEV, generator=_gen(seed + 1)) < case["solid"]).cpu()
        force = (1e-6, 0.0, 0.0)
    elif case["kind"] == "droplet":
        x, y, z = _grid(shape)
        at = [n / 2 + float(torch.rand((), generator=r)) - 0.5 for n in (nx, ny, nz)]
        dist = ((x - at[0]) ** 2 + (y - at[1]) ** 2 + (z - at[2]) ** 2).sqrt()
        phi = 0.5 * (1 + torch.tanh(2 * (0.16 * min(shape) - dist) / 4.0))
        two = dict(rho_l=1.0, rho_h=1.0, tau_l=case["tau"], tau_h=case["tau"], sigma=0.03, width=4.0, diffusivity=0.1)
    elif case["kind"] == "layered":
        x, _, _ = _grid(shape)
        at = nx / 2 + float(torch.rand((), generator=r)) - 0.5
        phi = (0.5 * (1 + torch.tanh(2 * (x - at) / 4.0))).expand(shape).contiguous()
        mask = torch.zeros(shape, dtype=torch.bool)
        mask[..., 0] = mask[..., -1] = True
        two = dict(rho_l=0.5, rho_h=1.5, tau_l=case["tau"], tau_h=case["tau"] + 1.05, sigma=0.03, width=4.0, diffusivity=0.1,
                   body_accel=(0.0, 1e-7, 0.0))
    if case["storage"] == "f64":
        M = M.double()
    return M, mask, phi, two, force


def _adjoint_inputs(case, seed):
    """Force field on the fluid and target velocity of an adjoint case."""
    shape = (case["nz"], case["ny"], case["nx"])
    fluid = torch.ones(shape, device=DEV)
    fluid[:, 0] = fluid[:, -1] = 0.0
    F = torch.randn((3,) + shape, device=DEV, generator=_gen(seed + 70)) * 1e-6 * fluid
    target = torch.randn((3,) + shape, device=DEV, generator=_gen(seed + 71)) * 1e-4
    return F, target, fluid


def _loss(M, target, fluid):
    return (((M[1:4] - target) * fluid) ** 2).sum() / fluid.sum()


# --------------------------------------------------------------------------------------- a pass
def prepare(case, seed):
    M, mask, phi, two, force = _inputs(case, seed)
    shape = tuple(M.shape[1:])
    kw = dict(lattice=case["lattice"], tau=case["tau"], storage=case["storage"], mask=mask, device=DEV)
    if case["kind"] == "adjoint":
        F, target, fluid = _adjoint_inputs(case, seed)
        s = Solver(shape, force_field=F, **kw)
        return dict(case=case, solver=s, F=F.requires_grad_(True), M0=M.requires_grad_(True), target=target, fluid=fluid)
    s = Solver(shape, force=force, two_component=two, **kw)
    s.set_moments(M, phi)
    out = torch.empty_like(M)
    return dict(case=case, solver=s, out=out, sums=torch.empty(6, dtype=torch.float64, device=DEV),
                phi_out=None if phi is None else torch.empty_like(phi), load=(M, phi) if case["restart"] else None)


def run(st):
    case, s = st["case"], st["solver"]
    if case["kind"] == "adjoint":
        MT = rollout(st["F"], st["M0"], s, case["steps"], case["every"])
        gF, gM = torch.autograd.grad(_loss(MT, st["target"], st["fluid"]), (st["F"], st["M0"]))
        return {"moments": MT.detach(), "grad_force": gF, "grad_moments": gM}
    if st["load"] is not None:
        s.set_moments(*st["load"])
    s.step(case["steps"])
    s.reduce_async(st["sums"])
    M = s.moments(out=st["out"], phi_out=st["phi_out"])
    # 16-bit runs keep their snapshots in the type they store; sums are kept at the flow's precision
    got = {"moments": M.to(STORED[case["storage"]]), "sums": st["sums"].to(M.dtype)}
    if st["phi_out"] is not None:
        got["phi"] = st["phi_out"]
    return got


def work(case):
    n, b = case["nx"] * case["ny"] * case["nz"], BYTES[case["storage"]]
    site = 20 * b  # the 10 stored moments read and written
    flops = {"19": 300, "27": 420, "27h": 700}[case["lattice"]]
    if case["kind"] in ("channel", "porous", "layered", "adjoint"):
        site += 1  # mask
    if case["kind"] == "adjoint":
        # forward with its force field, the recomputed forward, and the adjoint step: cotangent in
        # and out (80), both velocities (24), force (12), mask, FP64 force gradient updated (48)
        return {"bytes": float(n * case["steps"] * (2 * (site + 12) + 165)), "flops": float(n * case["steps"] * 3 * flops)}
    if case["kind"] in ("droplet", "layered"):
        site += 8  # phase field read and written
        flops += 250
    out = 10 * (b + max(b, 4))
    load = 10 * (b + max(b, 4)) if case["restart"] else 0
    return {"bytes": float(n * (case["steps"] * site + out + load)), "flops": float(n * case["steps"] * flops)}


# ------------------------------------------------------------------------------ 64-bit reference
def _directions(lattice):
    got = []
    for c in [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]:
        n = sum(abs(v) for v in c)
        if lattice == "19" and n < 3:
            got.append((c, (1 / 3, 1 / 18, 1 / 36)[n]))
        elif lattice != "19":
            got.append((c, (8 / 27, 2 / 27, 1 / 54, 1 / 216)[n]))
    return got


def _roll(f, c):
    """The value at x - c, for every x."""
    return f if c == (0, 0, 0) else torch.roll(f, (c[2], c[1], c[0]), (0, 1, 2))


class _Collided:
    """Post-collision populations of moments M with force F (list of 3), density rho and rate omega."""

    def __init__(self, M, F, rho, omega, full):
        u = [M[1], M[2], M[3]]
        h = [f / (2 * rho) for f in F]
        keep = 1 - omega
        self.full, self.p, self.u, self.h = full, M[0], u, h
        self.N = [M[4 + i] - u[a] * u[b] for i, (a, b) in enumerate(SYM)]
        if full:
            self.N = [keep * n for n in self.N]
            return
        P = [u[a] * u[b] + keep * self.N[i] + u[a] * h[b] + h[a] * u[b] for i, (a, b) in enumerate(SYM)]
        self.b = [3 * (u[a] + h[a]) for a in range(3)]
        self.q0 = M[0] - 1.5 * (P[0] + P[1] + P[2])
        self.e = [(4.5 if a == b else 9.0) * P[i] for i, (a, b) in enumerate(SYM)]

    def population(self, c, w):
        if self.full:
            return self._product(c) * w
        f = self.q0.clone()
        for a in range(3):
            if c[a]:
                f.add_(self.b[a], alpha=c[a])
        for i, (a, b) in enumerate(SYM):
            if c[a] * c[b]:
                f.add_(self.e[i], alpha=c[a] * c[b])
        return f.mul_(w)

    def _product(self, c):
        """Complete basis: per axis 1 + 3 c u + 4.5 (c^2 - 1/3) u^2 and its derivatives in u."""
        k = [4.5 * (v * v - 1 / 3) for v in c]
        ps = [3.0 * c[a] * self.u[a] + k[a] * self.u[a] ** 2 for a in range(3)]
        ph = [1 + v for v in ps]
        dl = [3.0 * c[a] + 2 * k[a] * self.u[a] for a in range(3)]
        f = self.p + ps[0] + ph[0] * (ps[1] + ph[1] * ps[2])
        for a in range(3):
            f += self.h[a] * dl[a] * ph[(a + 1) % 3] * ph[(a + 2) % 3]
        for i, (a, b) in enumerate(SYM):
            if a == b:
                f += self.N[i] * k[a] * ph[(a + 1) % 3] * ph[(a + 2) % 3]
            else:
                f += self.N[i] * dl[a] * dl[b] * ph[3 - a - b]
        return f


def _stream(lattice, col, solid):
    """Raw moments [a0, a1 (3), a2 (6)] of the streamed populations, halfway bounce-back at solids."""
    acc = [torch.zeros_like(col.p) for _ in range(10)]
    for c, w in _directions(lattice):
        f = _roll(col.population(c, w), c)
        if solid is not None and c != (0, 0, 0):
            f = torch.where(_roll(solid, c), col.population(tuple(-v for v in c), w), f)
        acc[0].add_(f)
        for a in range(3):
            if c[a]:
                acc[1 + a].add_(f, alpha=c[a])
        for i, (a, b) in enumerate(SYM):
            if c[a] * c[b]:
                acc[4 + i].add_(f, alpha=c[a] * c[b])
    third = acc[0] / 3
    for i in range(3):
        acc[4 + i] = acc[4 + i] - third
    return acc


def _corrected(raw, F, rho):
    h = [f / (2 * rho) for f in F]
    u = [raw[1 + a] + h[a] for a in range(3)]
    return [raw[0]] + u + [raw[4 + i] + u[a] * h[b] + h[a] * u[b] for i, (a, b) in enumerate(SYM)]


def _held(new, old, solid):
    return new if solid is None else [torch.where(solid, o, n) for n, o in zip(new, old)]


def _stencils(psi):
    """Gradient (list of 3) and Laplacian of psi with the D3Q27 weights."""
    g, lap = [torch.zeros_like(psi) for _ in range(3)], torch.zeros_like(psi)
    for c, w in _directions("27"):
        v = _roll(psi, tuple(-k for k in c))
        lap.add_(v - psi, alpha=6 * w)
        for a in range(3):
            if c[a]:
                g[a].add_(v, alpha=3 * w * c[a])
    return g, lap


def _divergence(V):
    d = torch.zeros_like(V[0])
    for c, w in _directions("27"):
        for a in range(3):
            if c[a]:
                d.add_(_roll(V[a], tuple(-k for k in c)), alpha=3 * w * c[a])
    return d


class _Phases:
    """The two-component parts: blending, interface advance and the split force."""

    def __init__(self, two):
        self.t = two

    def rho(self, phi):
        return self.t["rho_l"] + phi * (self.t["rho_h"] - self.t["rho_l"])

    def nu(self, phi):
        return (self.t["tau_l"] - 0.5) / 3 + phi * ((self.t["tau_h"] - self.t["tau_l"]) / 3)

    def omega(self, phi):
        return 1 / (3 * self.nu(phi) + 0.5)

    def force(self, phi, p, neq):
        t = self.t
        g, lap = _stencils(phi)
        mu = 48 * t["sigma"] / t["width"] * phi * (phi - 1) * (phi - 0.5) - 1.5 * t["sigma"] * t["width"] * lap
        a = t.get("body_accel", (0.0, 0.0, 0.0))
        F = [mu * g[k] + self.rho(phi) * a[k] for k in range(3)]
        if t["rho_l"] != t["rho_h"]:
            gr = [v * (t["rho_h"] - t["rho_l"]) for v in g]
            S = [[neq[SYM.index((min(a, b), max(a, b)))] for b in range(3)] for a in range(3)]
            coef = -3 * self.nu(phi) * self.omega(phi)
            F = [F[a] - p / 3 * gr[a] + coef * sum(S[a][b] * gr[b] for b in range(3)) for a in range(3)]
        return F

    def advance(self, phi, u, solid):
        g, lap = _stencils(phi)
        size = torch.clamp((g[0] ** 2 + g[1] ** 2 + g[2] ** 2).sqrt(), min=1e-12)
        lam = 4 * self.t["diffusivity"] / self.t["width"]
        if solid is not None:
            u = [torch.where(solid, torch.zeros_like(v), v) for v in u]
        new = phi - _divergence([phi * u[a] + lam * phi * (1 - phi) * g[a] / size for a in range(3)]) + self.t["diffusivity"] * lap
        return new if solid is None else torch.where(solid, phi, new)


def _exact_two(case, M, phi, solid, two):
    ph = _Phases(two)
    F = ph.force(phi, M[0], [M[4 + i] - M[1 + a] * M[1 + b] for i, (a, b) in enumerate(SYM)])
    for _ in range(case["steps"]):
        new = ph.advance(phi, M[1:4], solid)
        raw = _stream(case["lattice"], _Collided(M, F, ph.rho(phi), ph.omega(phi), False), solid)
        phi = new
        F = ph.force(phi, raw[0], [raw[4 + i] - raw[1 + a] * raw[1 + b] for i, (a, b) in enumerate(SYM)])
        M = _held(_corrected(raw, F, ph.rho(phi)), M, solid)
    return M, phi


def _exact_adjoint(case, M, solid, seed):
    F, target, fluid = (t.double() for t in _adjoint_inputs(case, seed))
    F.requires_grad_(True)
    M0 = torch.stack(M).requires_grad_(True)
    parts = [F[a] for a in range(3)]

    def segment(n, *M):
        M = list(M)
        for _ in range(n):
            raw = _stream(case["lattice"], _Collided(M, parts, 1.0, 1 / case["tau"], False), solid)
            M = _held(_corrected(raw, parts, 1.0), M, solid)
        return tuple(M)

    now, left = tuple(M0[k] for k in range(10)), case["steps"]
    while left > 0:
        n = min(25, left)
        now, left = torch.utils.checkpoint.checkpoint(segment, n, *now, use_reentrant=False), left - n
    MT = torch.stack(now)
    gF, gM = torch.autograd.grad(_loss(MT, target, fluid), (F, M0))
    return {"moments": MT.detach(), "grad_force": gF, "grad_moments": gM}


def exact(case, seed):
    M, mask, phi, two, force = _inputs(case, seed)
    solid = None if mask is None else mask.to(DEV)
    M = [M[k].double() for k in range(10)]
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, M, solid, seed)
    if two is not None:
        M, phi = _exact_two(case, M, phi.double(), solid, two)
    else:
        F = [torch.tensor(f, dtype=torch.float64, device=DEV) for f in force]
        for _ in range(case["steps"]):
            raw = _stream(case["lattice"], _Collided(M, F, 1.0, 1 / case["tau"], case["lattice"] == "27h"), solid)
            M = _held(_corrected(raw, F, 1.0), M, solid)
    live = slice(None) if solid is None else ~solid
    sums = [M[k][live].sum() for k in range(4)] + [phi[live].sum() if phi is not None else M[0].new_zeros(())]
    sums.append(sum((M[1 + a][live] ** 2).sum() for a in range(3)))
    got = {"moments": torch.stack(M), "sums": torch.stack(sums)}
    if phi is not None:
        got["phi"] = phi
    return got
