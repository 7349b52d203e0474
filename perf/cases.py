"""What a user of the coupled step has it do, as timed cases.

One case is one kind of run (3D or 2D ripening, the diffusion couple, sedimentation with
flow, the diagnostics, the adjoint gradient) at one size, storage and option set. ``run``
takes it through the public classes: ``Simulation.step`` followed by ``Simulation.fields``,
as a run that writes its fields every few steps does, ``Simulation.sums``, and
``adjoint.misfit_and_gradient``. A simulation goes on from where the last pass left it.
``exact`` is the same scheme in plain torch in FP64.
"""
import math

import torch

from paper_2409_03401_gb300 import Simulation
from paper_2409_03401_gb300.adjoint import misfit_and_gradient
from workloads.configs import (LAMBDA_COUPLE, M_PHI_COUPLE, RIPENING_2D_M, RIPENING_2D_M_PHI, RIPENING_2D_R,
                               SUPERSATURATION, THETA_EVAL, with_theta)
from workloads.params import LBMParams

SCALARS = ("phi", "muA", "muB")
FLOW = ("phi", "muA", "muB", "p", "ux", "uy", "uz")
# the sum of p_h is an invariant whose value is 0: only its rounding would come back
SUMS = ("phi", "cA", "cB", "S", "umax", "g", "nonfinite", "interface", "euler")


def _case(name, kind, nx, ny, nz, steps, lattice="D3Q7", storage="f32", collision="BGK", inplace=False, walls=True,
          every=0):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "steps": steps, "lattice": lattice, "storage": storage,
         "collision": collision, "inplace": inplace, "walls": walls, "every": every}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the 2D diffusion couple at its full size, FP64: 4096 nodes, every step is one small launch
        _case("couple 512x8 f64", "couple", 512, 8, 1, 100, lattice="D2Q5", storage="f64"),
        # the reduced-size 3D ripening run, 20,000 steps long in earnest: launches count
        _case("ripening 48^3", "ripening", 48, 48, 48, 100),
        # the 3D ripening workload, no flow, periodic
        _case("ripening 256^3", "ripening", 256, 256, 256, 20),
        # the 2D ripening workload on D2Q9, the largest 2D lattice
        _case("ripening 2D 4096^2", "ripening2d", 4096, 4096, 1, 20, lattice="D2Q9"),
        # the reduced-size sedimentation run with flow: a lattice too small to fill the chip by itself
        _case("sedimentation 64^3", "flow", 64, 64, 64, 50),
        # the sedimentation workload: the largest lattice, the case the framework exists for
        _case("sedimentation 512^3", "flow", 512, 512, 512, 20),
        # the drift study with 16-bit storage, two state copies
        _case("drift 384^3 f16", "flow", 384, 384, 384, 10, storage="f16"),
        # 16-bit storage in the in-place layout, for the least memory
        _case("sedimentation 256^3 f16 in place", "flow", 256, 256, 256, 20, storage="f16", inplace=True),
        # an odd box with the MRT collision
        _case("sedimentation 251x190x131 MRT", "flow", 251, 190, 131, 10, collision="MRT"),
        # the paper's choice of D3Q19 for every equation
        _case("sedimentation 192^3 D3Q19", "flow", 192, 192, 192, 10, lattice="D3Q19"),
        # the diagnostics that a long run logs: sums, max |u|, interface, droplet count
        _case("diagnostics 384^3", "sums", 384, 384, 384, 4),
        # misfit and gradient of the parameter-estimation workload, checkpoints in the proportion of its own
        _case("adjoint 128^3", "adjoint", 128, 128, 128, 40, every=20),
    ]


def _size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    # half of the extents are multiples of 16, as users like them; the others come as they fall, odd ones too
    return max(16, (n + 8) // 16 * 16) if rng.random() < 0.5 else n


def _box(rng, lo, hi, most):
    while True:
        n = [_size(rng, lo, hi) for _ in range(3)]
        if n[0] * n[1] * n[2] <= most:
            return n


def draw(rng):
    kind = rng.choice(["couple", "ripening", "ripening", "ripening2d", "flow", "flow", "flow", "sums", "adjoint"])
    steps = 2 * rng.randint(3, 15)
    if kind == "couple":
        return _case(None, kind, _size(rng, 64, 2048), rng.randint(4, 40), 1, 4 * steps, lattice="D2Q5", storage="f64")
    if kind == "ripening2d":
        return _case(None, kind, _size(rng, 200, 4000), _size(rng, 200, 4000), 1, steps, lattice="D2Q9",
                     storage=rng.choice(["f32", "f32", "f64"]))
    if kind == "ripening":
        nx, ny, nz = _box(rng, 32, 288, 2 ** 24)
        return _case(None, kind, nx, ny, nz, steps, storage=rng.choice(["f32", "f32", "f32", "f64", "f16"]),
                     lattice=rng.choice(["D3Q7", "D3Q7", "D3Q7", "D3Q19"]))
    if kind == "adjoint":
        nx, ny, nz = _box(rng, 24, 128, 2 ** 21)
        return _case(None, kind, nx, ny, nz, steps, every=rng.randint(4, steps))
    nx, ny, nz = _box(rng, 32, 400, 2 ** 25)
    storage = rng.choice(["f32", "f32", "f32", "f16", "f16", "bf16", "f64"])
    if storage == "f64":
        nx, ny, nz = _box(rng, 32, 160, 2 ** 21)
    lattice = "D3Q19" if storage == "f32" and rng.random() < 0.25 else "D3Q7"
    return _case(None, kind, nx, ny, nz, steps if kind == "flow" else 4, lattice=lattice, storage=storage,
                 collision=rng.choice(["BGK", "BGK", "TRT", "MRT"]), inplace=rng.random() < 0.3,
                 walls=rng.random() < 0.75)


def _params(c):
    flow = c["kind"] in ("flow", "sums")
    size = dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], lattice=c["lattice"], storage=c["storage"])
    if c["kind"] == "couple":
        return LBMParams(wall_x=True, lam=LAMBDA_COUPLE, M_phi=M_PHI_COUPLE, c_eq=((0.1, 0.3), (0.6, 0.1)),
                         M=((0.5, 0.5), (1.0, 1.0)), **size)
    if c["kind"] == "ripening2d":
        return LBMParams(M_phi=RIPENING_2D_M_PHI, M=(RIPENING_2D_M, RIPENING_2D_M), **size)
    p = LBMParams(flow=flow, wall_z=flow and c["walls"], inplace=c["inplace"], collision=c["collision"], **size)
    return with_theta(p, THETA_EVAL) if c["kind"] == "adjoint" else p


def _droplets(c, gen, r_min, r_max, dev):
    """phi of one droplet per cell of a grid over the box, at a random place in its cell and of
    a random radius that fits it."""
    n = (c["nz"], c["ny"], c["nx"])
    cells = [max(1, int(m // (2 * r_max + 6))) for m in n]
    room = [1e9 if m == 1 else m / k for m, k in zip(n, cells)]
    fit = max(1.5, min(r_max, min(room) / 2 - 1.5))
    rand = torch.rand(cells + [4], generator=gen, device=dev, dtype=torch.float64)
    r = min(r_min, 0.6 * fit) + (fit - min(r_min, 0.6 * fit)) * rand[..., 3]
    at = [torch.arange(m, device=dev) for m in n]
    which = [(a * k) // m for a, k, m in zip(at, cells, n)]
    which = which[0][:, None, None], which[1][None, :, None], which[2][None, None, :]
    d2 = 0.0
    for ax in range(3):
        if n[ax] == 1:
            continue
        size = n[ax] / cells[ax]
        start = torch.arange(cells[ax], device=dev, dtype=torch.float64).reshape([-1 if i == ax else 1 for i in range(3)])
        centre = size * start + r + 1 + (size - 2 * r - 2).clamp(min=0.0) * rand[..., ax]
        x = at[ax].to(torch.float64).reshape([-1 if i == ax else 1 for i in range(3)])
        d2 = d2 + (x - centre[which]) ** 2
    return 0.5 * (1.0 + torch.tanh((r[which] - torch.sqrt(d2)) * (2.0 / 3.0)))


def _inputs(c, seed, dev="cuda"):
    p = _params(c)
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    if c["kind"] == "couple":
        # a planar interface with a little waviness along y, phase 1 on its left
        y = torch.arange(c["ny"], device=dev, dtype=torch.float64)[None, :, None]
        x = torch.arange(c["nx"], device=dev, dtype=torch.float64)[None, None, :]
        a = torch.rand(2, generator=gen, device=dev, dtype=torch.float64)
        xi = c["nx"] / 2 - 0.5 + 4 * (a[0] - 0.5) + a[1] * torch.cos(2 * math.pi * y / c["ny"])
        phi = 0.5 * (1.0 - torch.tanh((x - xi) * (2.0 / p.W)))
        inside, outside = (0.55, 0.15), (0.15, 0.25)
    else:
        lo, hi = RIPENING_2D_R if c["kind"] == "ripening2d" else (6.0, 16.0) if p.flow else (4.0, 10.0)
        phi = _droplets(c, gen, lo, hi, dev)
        d = 0.1 if c["kind"] == "ripening2d" else SUPERSATURATION
        inside = p.c_eq[1]
        outside = tuple((1 - d) * p.c_eq[0][a] + d * p.c_eq[1][a] for a in range(2))
    cA, cB = (torch.where(phi >= 0.5, inside[a], outside[a]).to(torch.float64) for a in range(2))
    return p, phi.contiguous(), cA.contiguous(), cB.contiguous()


def _target(c, seed, dev="cuda"):
    """The observed fields of the gradient: other droplets, and mu near its initial values."""
    p, phi, cA, cB = _inputs(c, seed + 7919, dev)
    return tuple(t.to(torch.float32) for t in (phi, 1e-3 * (1 + phi), 1e-3 * (1 - phi)))


def prepare(case, seed):
    p, phi, cA, cB = _inputs(case, seed)
    if case["kind"] == "adjoint":
        return {"case": case, "p": p, "in": (phi, cA, cB), "target": _target(case, seed)}
    sim = Simulation(p, phi, cA, cB, device="cuda")
    if case["kind"] == "sums":
        sim.step(case["steps"])
    return {"case": case, "sim": sim}


def run(state):
    c = state["case"]
    if c["kind"] == "adjoint":
        L, gtheta, gphi = misfit_and_gradient(state["p"], THETA_EVAL, *state["in"], c["steps"], state["target"],
                                              K=c["every"])
        return {"L": L, "dtheta": gtheta, "dphi0": gphi}
    sim = state["sim"]
    if c["kind"] == "sums":
        s = sim.sums()
        return {k: s[k] for k in SUMS}
    return sim.step(c["steps"]).fields(FLOW if c["kind"] == "flow" else SCALARS)


def work(case):
    # bytes: the state read once and written once a pass, and the fields written; flops: every step's
    # arithmetic of the scheme (moments, closure, stencil and collisions, counted from its equations)
    p = _params(case)
    q = {"D2Q5": 5, "D2Q9": 9, "D3Q7": 7, "D3Q19": 19}[case["lattice"]]
    pops = 3 * q + (19 if p.flow else 0)
    size = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[case["storage"]]
    rest = (4 if p.flow else 3) * 2 if size == 2 else 0       # rest populations of 16-bit storage are FP32
    real = 8 if size == 8 else 4
    n = float(p.nodes)
    step_flops = 3 * q * 8 + 60 + (19 * 24 + 160 if p.flow else 0)
    if case["kind"] == "sums":
        return {"bytes": n * (pops * size + rest), "flops": n * (3 * q + 60 + (240 if p.flow else 0))}
    if case["kind"] == "adjoint":
        # each step forward, again from the checkpoints, and its transpose
        return {"bytes": n * 8 * (3 + 1 + 3), "flops": n * case["steps"] * 4 * step_flops}
    fields = len(FLOW) if p.flow else len(SCALARS)
    return {"bytes": n * (2 * (pops * size + rest) + fields * real), "flops": n * case["steps"] * step_flops}


# ---------------------------------------------------------------------------------------
# The scheme in plain torch, FP64: populations are lists of (nz, ny, nx) tensors.
_AXES = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
_EDGES = [(a, b, 0) for a in (1, -1) for b in (1, -1)] + [(a, 0, b) for a in (1, -1) for b in (1, -1)] + \
    [(0, a, b) for a in (1, -1) for b in (1, -1)]
_SETS = {
    "D2Q5": (_AXES[:5], [1 / 3] + [1 / 6] * 4, 1 / 3),
    "D2Q9": (_AXES[:5] + _EDGES[:4], [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, 1 / 3),
    "D3Q7": (_AXES, [1 / 4] + [1 / 8] * 6, 1 / 4),
    "D3Q19": (_AXES + _EDGES, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, 1 / 3),
}
_E19, _W19, _ = _SETS["D3Q19"]
_OPP19 = [_E19.index((-e[0], -e[1], -e[2])) for e in _E19]


def _dot(e, v):
    s = None
    for ek, vk in zip(e, v):
        if ek:
            t = vk if ek > 0 else -vk
            s = t if s is None else s + t
    return 0.0 if s is None else s


class _Exact:
    def __init__(self, p, theta=None):
        self.p = p
        self.e, self.w, self.cs2 = _SETS[p.lattice]
        self.M, self.M_phi = p.M, p.M_phi
        if theta is not None:
            self.M, self.M_phi = ((theta[0],) * 2, (theta[1],) * 2), theta[2]

    def mu(self, c, phi, a):
        pp = phi * phi * (3 - 2 * phi)
        return c - (1 - pp) * self.p.c_eq[0][a] - pp * self.p.c_eq[1][a]

    def source(self, phi, cA, cB):
        p = self.p
        dom = sum(self.mu(c, phi, a) * (p.c_eq[1][a] - p.c_eq[0][a]) for a, c in ((0, cA), (1, cB)))
        return self.M_phi / p.W ** 2 * (-16 * phi * (1 - phi) * (1 - 2 * phi) + p.lam * 6 * phi * (1 - phi) * dom)

    def force(self, phi):
        """Capillary force and buoyancy; the walled component of a step beyond a wall is dropped."""
        p = self.p
        g, lap = [0.0, 0.0, 0.0], 0.0
        for e, w in zip(_E19[1:], _W19[1:]):
            nb = torch.roll(phi, (-e[2], -e[1], -e[0]), (0, 1, 2))
            if p.wall_z and e[2]:
                edge = -1 if e[2] > 0 else 0
                nb[edge] = torch.roll(phi[edge], (-e[1], -e[0]), (0, 1))
            for a in range(3):
                if e[a]:
                    g[a] = g[a] + 3 * w * e[a] * nb
            lap = lap + 6 * w * (nb - phi)
        br = 1.5 * p.sigma * p.W * (16 * phi * (1 - phi) * (1 - 2 * phi) / p.W ** 2 - lap)
        return [br * g[a] + phi * p.g[a] for a in range(3)]

    def start(self, phi, cA, cB):
        S = self.source(phi, cA, cB)
        muA, muB = self.mu(cA, phi, 0), self.mu(cB, phi, 1)
        self.g = [w * phi - w * S / 2 for w in self.w]
        self.h = [[c - (1 - self.w[0]) * m if k == 0 else w * m for k, w in enumerate(self.w)]
                  for c, m in ((cA, muA), (cB, muB))]
        if self.p.flow:
            F = self.force(phi)
            self.f = [-0.5 * w * _dot(e, F) + torch.zeros_like(phi) for e, w in zip(_E19, _W19)]
        return self

    def moments(self):
        cA, cB, phit = sum(self.h[0]), sum(self.h[1]), sum(self.g)
        S = self.source(phit, cA, cB)
        phi = phit + S / 2
        out = {"phi": phi, "muA": self.mu(cA, phi, 0), "muB": self.mu(cB, phi, 1), "cA": cA, "cB": cB, "S": S,
               "g": phit}
        if self.p.flow:
            F = self.force(phi)
            u = [3 * sum(e[a] * f for e, f in zip(_E19, self.f) if e[a]) + F[a] / 2 for a in range(3)]
            out |= {"p": sum(self.f), "ux": u[0], "uy": u[1], "uz": u[2], "F": F}
        return out

    def stream(self, post, e):
        p, opp = self.p, [e.index((-x, -y, -z)) for x, y, z in e]
        new = list(post)
        for k, (x, y, z) in enumerate(e):
            if k == 0:
                continue
            new[k] = torch.roll(post[k], (z, y, x), (0, 1, 2))
            if p.wall_z and z:
                new[k][0 if z > 0 else -1] = post[opp[k]][0 if z > 0 else -1]
            if p.wall_x and x:
                new[k][:, :, 0 if x > 0 else -1] = post[opp[k]][:, :, 0 if x > 0 else -1]
        return new

    def step(self):
        p, m = self.p, self.moments()
        phi, S = m["phi"], m["S"]
        u = [m["ux"], m["uy"], m["uz"]] if p.flow else None
        om = 1 / (self.M_phi / self.cs2 + 0.5)
        cu = [_dot(e, u) / self.cs2 if u else 0.0 for e in self.e]
        for a, (c, mu) in enumerate(((m["cA"], m["muA"]), (m["cB"], m["muB"]))):
            rate = 1 / ((self.M[0][a] * (1 - phi) + self.M[1][a] * phi) / self.cs2 + 0.5)
            for k, w in enumerate(self.w):
                eq = c - (1 - w) * mu if k == 0 else w * mu + w * c * cu[k]
                self.h[a][k] = self.h[a][k] - rate * (self.h[a][k] - eq)
            self.h[a] = self.stream(self.h[a], self.e)
        self.g = self.stream([g - om * (g - w * phi * (1 + x) + w * S / 2) + w * S
                              for g, w, x in zip(self.g, self.w, cu)], self.e)
        if p.flow:
            self.flow(m, u)

    def flow(self, m, u):
        p, F = self.p, m["F"]
        om = 1 / (3 * p.nu + 0.5)
        usq, uF = sum(v * v for v in u), sum(a * b for a, b in zip(u, F))

        def off(k):
            """f_k - f_k^eq, and F_k"""
            cu = _dot(_E19[k], u)
            Fk = _W19[k] * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq) * (_dot(_E19[k], F) - uF)
            return self.f[k] - _W19[k] * (m["p"] + cu + 1.5 * cu * cu - 0.5 * usq) + Fk / 2, Fk

        if p.collision == "MRT":
            d, Fk = zip(*(off(k) for k in range(19)))
            relax = torch.einsum("kl,lzyx->kzyx", _mrt(p, om, d[0].device), torch.stack(d))
            post = [f - r + x for f, r, x in zip(self.f, relax, Fk)]
        else:
            other = 1 / (p.trt_magic / (1 / om - 0.5) + 0.5) if p.collision == "TRT" else om
            post = list(self.f)
            for k in range(19):
                if _OPP19[k] < k:
                    continue
                (a, Fa), (b, Fb) = off(k), off(_OPP19[k])
                even, odd = om * (a + b) / 2, other * (a - b) / 2
                post[k] = self.f[k] - even - odd + Fa
                if _OPP19[k] != k:
                    post[_OPP19[k]] = self.f[_OPP19[k]] - even + odd + Fb
        self.f = self.stream(post, _E19)


def _mrt(p, om, dev):
    """M^-1 S M on d'Humieres' orthogonal basis of D3Q19."""
    rows, (se, seps, sq, spi, sm) = [], p.mrt_rates
    for x, y, z in _E19:
        c = x * x + y * y + z * z
        xx, ww = 3 * x * x - c, y * y - z * z
        rows.append([1, 19 * c - 30, (21 * c * c - 53 * c + 24) / 2, x, (5 * c - 9) * x, y, (5 * c - 9) * y, z,
                     (5 * c - 9) * z, xx, (3 * c - 5) * xx, ww, (3 * c - 5) * ww, x * y, y * z, x * z, ww * x,
                     (z * z - x * x) * y, (x * x - y * y) * z])
    M = torch.tensor(rows, dtype=torch.float64, device=dev).T
    s = torch.tensor([om, se, seps, om, sq, om, sq, om, sq, om, spi, om, spi, om, om, om, sm, sm, sm],
                     dtype=torch.float64, device=dev)
    return M.T @ torch.diag(s / (M * M).sum(1)) @ M


def _euler(on, wall_z):
    """Vertices - edges + faces - cubes of the union of closed unit cubes on the set nodes."""
    b = torch.nn.functional.pad(on.to(torch.uint8), (0, 0, 0, 0, 1, 1)).bool() if wall_z else on

    def low(t, axes):
        for a in axes:
            t = t | torch.roll(t, 1, a)
        return t
    return sum((-1) ** (3 - len(axes)) * int(low(b, axes).sum())
               for axes in ((), (0,), (1,), (2,), (0, 1), (0, 2), (1, 2), (0, 1, 2)))


def exact(case, seed):
    p, phi, cA, cB = _inputs(case, seed)
    if case["kind"] == "adjoint":
        return _exact_gradient(case, seed, p, phi, cA, cB)
    if p.nodes * case["steps"] > 3e9:
        return None
    with torch.no_grad():
        ex = _Exact(p).start(phi, cA, cB)
        for _ in range(case["steps"]):
            ex.step()
        m = ex.moments()
        if case["kind"] != "sums":
            return {k: m[k] for k in (FLOW if p.flow else SCALARS)}
        f = m["phi"]
        return {"phi": float(f.sum()), "cA": float(m["cA"].sum()), "cB": float(m["cB"].sum()),
                "S": float(m["S"].sum()), "g": float(m["g"].sum()), "nonfinite": 0.0,
                "umax": float((m["ux"] ** 2 + m["uy"] ** 2 + m["uz"] ** 2).max().sqrt()),
                "interface": float((4 / p.W * f * (1 - f)).sum()), "euler": float(_euler(f >= 0.5, p.wall_z))}


def _exact_gradient(case, seed, p, phi, cA, cB):
    from torch.utils.checkpoint import checkpoint
    th = torch.tensor(THETA_EVAL, dtype=torch.float64, device=phi.device, requires_grad=True)
    phi = phi.clone().requires_grad_(True)
    q = len(_SETS[p.lattice][1])

    def one(theta, *pops):
        ex = _Exact(p, theta)
        ex.g, ex.h = list(pops[:q]), [list(pops[q:2 * q]), list(pops[2 * q:])]
        ex.step()
        return (*ex.g, *ex.h[0], *ex.h[1])
    ex = _Exact(p, th).start(phi, cA, cB)
    pops = (*ex.g, *ex.h[0], *ex.h[1])
    for _ in range(case["steps"]):
        pops = checkpoint(one, th, *pops, use_reentrant=False)
    ex.g, ex.h = list(pops[:q]), [list(pops[q:2 * q]), list(pops[2 * q:])]
    m = ex.moments()
    t = _target(case, seed)
    L = 0.5 * sum(((m[k] - x.double()) ** 2).sum() for k, x in zip(SCALARS, t))
    L.backward()
    return {"L": float(L.detach()), "dtheta": th.grad.cpu(), "dphi0": phi.grad}
