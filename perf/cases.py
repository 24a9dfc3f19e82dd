"""The work this library is measured on: its lattice Boltzmann steps and its
energy minimisation, called as a user's program calls them.

Every case is one kind of study of the Diffuse Solid Method with its sizes; the
sizes come from the workloads of ``bench.py``, ``synthetic`` and the tests, and
``draw`` spreads them over the ranges those stand for.  ``prepare`` makes the
inputs on the GPU from the seed (geometry, liquid, contact angle, noise),
``run`` is one pass (a few to a few hundred steps and the read of the result,
one energy and gradient, one run of the minimiser) and ``exact`` repeats the
pass in 64 bits with plain torch operations.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2504_19941_gb300 as P
from paper_2504_19941_gb300.energy import Energy, FreeEnergy, lbfgs
from paper_2504_19941_gb300.serving import GpuExecutor

DEV = "cuda"
PERIODIC = ("periodic",) * 6
MIRROR_Y = ("periodic", "periodic", "mirror", "mirror", "periodic", "periodic")
WIDTH3 = 3.0 / (2.0 * math.log(9.0))   # tanh width of a 10-90 % rise over 3 nodes


def listed():
    return [
        # a liquid slab on a micropillar array, FP32: the benchmark workload, a
        # long run whose state is read every 20 steps
        dict(name="slab", kind="slab", nx=256, ny=256, nz=192, steps=20),
        # one served wetting study in 3D from set-up to fields, odd sides
        dict(name="request", kind="request", nx=101, ny=101, nz=101, steps=100),
        # one quantum of the serving loop: small lattices batched, large ones
        # on streams of their own
        dict(name="served", kind="served", flat=5, solid=3, side=129, steps=64),
        # capillary rise between plates under gravity, FP16 storage, the largest
        dict(name="plates_f16", kind="plates", nx=384, ny=384, nz=256, steps=10),
        # gas of a fifth of the liquid's density and another viscosity, ragged
        dict(name="contrast", kind="contrast", nx=250, ny=130, nz=101, steps=20),
        # filling of an inclined channel, D2Q9, mirror faces, viscosity contrast
        dict(name="channel", kind="channel", nx=1750, ny=450, steps=100),
        # the relaxation of that channel's solid, which comes before it
        dict(name="relax", kind="relax", nx=1750, ny=450, steps=200),
        # a drop on a flat wall, D2Q9, FP64: the smallest lattice
        dict(name="drop_f64", kind="drop64", nx=128, ny=64, steps=100),
        # a row of pillars, D2Q9, FP32, a large lattice in two dimensions
        dict(name="row2d", kind="row2d", nx=4096, ny=4096, steps=10),
        # three fluids on the pillar array
        dict(name="three_fluids", kind="multi", nfluid=3, nx=256, ny=256, nz=192, steps=10),
        # free energy and its gradient through autograd, a drop on a wavy wall
        dict(name="energy", kind="energy", nx=128, ny=128, nz=128),
        # iterations of the energy minimiser on the same drop
        dict(name="lbfgs", kind="lbfgs", nx=128, ny=128, nz=128, iters=25),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["slab", "request", "served", "plates", "contrast", "channel", "relax",
                       "drop64", "row2d", "multi", "energy", "lbfgs"])
    c = dict(kind=kind)
    if kind in ("slab", "multi"):
        c.update(nx=_log_int(rng, 48, 256), ny=_log_int(rng, 48, 256), nz=_log_int(rng, 64, 192),
                 steps=rng.randint(8, 20 if kind == "slab" else 10))
        if kind == "multi":
            c.update(nfluid=rng.choice([2, 3, 3, 4]))
    elif kind == "request":
        side = _log_int(rng, 64, 160)
        c.update(nx=side, ny=side, nz=side, steps=rng.randint(50, 100))
    elif kind == "served":
        c.update(flat=rng.randint(2, 6), solid=rng.randint(0, 3), side=rng.randint(64, 144),
                 steps=rng.randint(32, 64))
    elif kind == "plates":
        c.update(nx=_log_int(rng, 160, 384), ny=_log_int(rng, 128, 384),
                 nz=_log_int(rng, 48, 256), steps=rng.randint(5, 10))
    elif kind == "contrast":
        c.update(nx=_log_int(rng, 40, 256), ny=_log_int(rng, 40, 256), nz=_log_int(rng, 64, 160),
                 steps=rng.randint(8, 20))
    elif kind in ("channel", "relax"):
        nx = _log_int(rng, 500, 1750)
        c.update(nx=nx, ny=_log_int(rng, 200, 450), steps=rng.randint(50, 100))
    elif kind == "drop64":
        nx = _log_int(rng, 64, 256)
        c.update(nx=nx, ny=_log_int(rng, 48, 128), steps=rng.randint(50, 100))
    elif kind == "row2d":
        c.update(nx=_log_int(rng, 400, 4096), ny=_log_int(rng, 300, 4096),
                 steps=rng.randint(5, 20))
    else:
        if rng.random() < 0.3:   # the two-dimensional critical-pressure boxes
            c.update(nx=_log_int(rng, 64, 320), ny=_log_int(rng, 100, 400), nz=1)
        else:
            c.update(nx=_log_int(rng, 32, 144), ny=_log_int(rng, 32, 144),
                     nz=_log_int(rng, 48, 144))
        if kind == "lbfgs":
            c.update(iters=rng.randint(10, 25))
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _coords(shape):
    """Node coordinates as FP64 tensors that broadcast to (nz, ny, nx) or (ny, nx)."""
    d = len(shape)
    out = []
    for a, n in enumerate(shape):
        v = [1] * d
        v[d - 1 - a] = n
        out.append(torch.arange(n, dtype=torch.float64, device=DEV).reshape(v))
    return out


def _pillars(shape, base, width, pitch, height, offset):
    """Signed distance to a base plate with rectangular pillars, positive inside."""
    X = _coords(shape)
    z, length = X[-1], shape[-1]
    dz = z - 0.5 * (base - 1)
    plate = 0.5 * base - (dz - length * torch.round(dz / length)).abs()
    q = [(z - (base + 0.5 * (height - 1))).abs() - 0.5 * height]
    for x in X[:-1]:
        dx = x - offset - 0.5 * (width - 1)
        q.append((dx - pitch * torch.round(dx / pitch)).abs() - 0.5 * width)
    q = torch.stack(torch.broadcast_tensors(*q))
    box = -(q.clamp(min=0).square().sum(0).sqrt() + q.amax(0).clamp(max=0))
    return torch.maximum(plate.expand_as(box), box).contiguous()


def _slab(x, lo, hi):
    """Nodes lo .. hi - 1 of a coordinate, as a tanh layer."""
    return 0.25 * (1 + torch.tanh((x - lo + 0.5) / 2)) * (1 + torch.tanh((hi - 0.5 - x) / 2))


def _noise(gen, shape, like):
    return 2e-3 * torch.rand(shape, generator=gen, device=DEV, dtype=like) - 1e-3


def _profile(sd, width):
    return 0.5 + 0.5 * torch.tanh(sd / (2.0 * width))


def _problem(case, seed):
    """What the study hands to the library: dict of its parameters and fields."""
    kind = case["kind"]
    rng = random.Random(seed)
    gen = _gen(seed)
    pr = dict(lattice="D3Q19", prec="f32", theta=rng.uniform(95.0, 145.0), g12=2.5e-3, g23=2.5e-3,
              alpha_s=WIDTH3, rho=(1.0, 1.0), tau=(1.0, 1.0), body=(0.0, 0.0, 0.0),
              faces=PERIODIC, stage=2)
    if kind in ("slab", "multi", "contrast"):
        shape = (case["nx"], case["ny"], case["nz"])
        sd = _pillars(shape, 8, 10, 32, 30, rng.randrange(32))
        c2 = _slab(_coords(shape)[2], 38, min(98, case["nz"] - 8)).expand(sd.shape)
        if kind == "contrast":
            pr.update(rho=(1.0, 0.2), tau=(1.0, 0.7))
        if kind == "slab":
            pr.update(body=(0.0, 0.0, -1e-7 * rng.uniform(0.5, 1.5)))
    elif kind == "request":
        shape = (case["nx"], case["ny"], case["nz"])
        pr.update(theta=rng.uniform(30.0, 150.0))
        sd, c2 = _request(shape, rng)
    elif kind == "plates":
        shape = (case["nx"], case["ny"], case["nz"])
        X = _coords(shape)
        gap, thick = 40, 8
        x0, x1 = 40, shape[0] - 44
        dy = (X[1] - 0.5 * (shape[1] - 1)).abs() - 0.5 * gap
        plate = torch.minimum(torch.minimum(X[0] - x0 + 0.5, x1 - 0.5 - X[0]),
                              torch.minimum(dy, thick - dy))
        lid = torch.maximum(7.5 - X[0], X[0] - (shape[0] - 8.5))
        sd = torch.maximum(plate, lid).expand(shape[::-1]).contiguous()
        c2 = _slab(X[0], 8, 60 + rng.randrange(12)).expand(sd.shape)
        pr.update(prec="f16", theta=45.0, g12=1e-2, g23=1e-2,
                  body=(-2.0 * 1e-2 * math.cos(math.radians(45.0)) / (120.0 * gap), 0.0, 0.0))
    elif kind in ("channel", "relax"):
        shape = (case["nx"], case["ny"])
        x, y = _coords(shape)
        a = math.radians(20.0)
        length = min(900.0, 0.55 * shape[0], (shape[1] - 100.0) / math.sin(a))
        xe, ye = 0.17 * shape[0] + rng.uniform(-8, 8), 0.16 * shape[1]
        s = (x - xe) * math.cos(a) + (y - ye) * math.sin(a)
        t = -(x - xe) * math.sin(a) + (y - ye) * math.cos(a)
        sd = torch.minimum(torch.minimum(s, length - s), t.abs() - 20.0).contiguous()
        c2 = 0.25 * (1 + torch.tanh((s + 0.1 * shape[0]) / 2)) * (1 - torch.tanh(s / 2))
        pr.update(lattice="D2Q9", theta=60.0, alpha_s=1.0, tau=(1.0, 0.52), faces=MIRROR_Y)
        if kind == "relax":
            pr.update(stage=1, tau=(1.0, 1.0))
    elif kind == "drop64":
        shape = (case["nx"], case["ny"])
        x, y = _coords(shape)
        dy = y - 3.5
        sd = (4.0 - (dy - shape[1] * torch.round(dy / shape[1])).abs()).expand(
            shape[::-1]).contiguous()
        r = ((x - shape[0] / 2.0) ** 2 + (y - 7.5) ** 2).sqrt()
        c2 = 0.5 * (1 + torch.tanh((0.39 * min(shape) - r) / 2))
        pr.update(lattice="D2Q9", prec="f64", theta=60.0, alpha_s=4.0 / (2.0 * math.log(9.0)))
    elif kind == "row2d":
        shape = (case["nx"], case["ny"])
        sd = _pillars(shape, 8, 10, 32, 30, rng.randrange(32))
        c2 = _slab(_coords(shape)[1], 38, 98).expand(sd.shape)
        pr.update(lattice="D2Q9")
    else:
        raise ValueError(kind)
    real = torch.float64 if pr["prec"] == "f64" else torch.float32
    c1 = _profile(sd, pr["alpha_s"])
    c2 = (c2 + _noise(gen, c2.shape, torch.float64)) * (1.0 - c1)
    pr.update(shape=shape, sd=sd.to(real).reshape(-1), c1=c1.to(real).reshape(-1),
              c2=c2.to(real).reshape(-1).contiguous(), real=real)
    if kind == "multi":
        nf = case["nfluid"] - 1
        C = [pr["c2"]]
        if nf >= 2:
            left = (torch.arange(pr["c2"].numel(), device=DEV) % shape[0] < shape[0] // 2).float()
            C = [pr["c2"] * left, pr["c2"] * (1 - left)]
        if nf == 3:
            z = (torch.arange(pr["c2"].numel(), device=DEV) // (shape[0] * shape[1]))
            C.append(((1 - pr["c1"] - pr["c2"]) * (z >= int(0.78 * shape[2]))).clamp(min=0))
        pr.update(C=torch.stack(C).contiguous())
    if kind == "relax":
        pr.update(mask=(sd > 0).to(torch.uint8).reshape(-1), beta=1e-3, omega=2e-4,
                  c1=(sd > 0).to(real).reshape(-1))
    return pr


def _request(shape, rng):
    """Geometry and drop of one served wetting study."""
    side, d = shape[0], len(shape)
    X = _coords(shape)
    if rng.randrange(2):
        pitch = rng.randint(16, 32)
        sd = _pillars(shape, 6, rng.randint(4, pitch // 2), pitch, rng.randint(8, side // 4), 0)
    else:
        k = 2 * math.pi / rng.uniform(16, 64)
        amp = rng.uniform(2, 8)
        slope = amp * k * torch.cos(k * X[0])
        sd = ((8.0 + amp * torch.sin(k * X[0]) - X[-1]) / (1 + slope * slope).sqrt()).expand(
            shape[::-1]).contiguous()
    centre = [s / 2.0 for s in shape]
    centre[-1] = side / 3.0
    r = sum((X[a] - centre[a]) ** 2 for a in range(d)).sqrt()
    return sd, 0.5 * (1 + torch.tanh((side / 5.0 - r) / 2))


def _params(pr):
    return P.make_params(pr["lattice"], pr["shape"], pr["prec"], theta_deg=pr["theta"],
                         g12=pr["g12"], g23=pr["g23"], alpha_s=pr["alpha_s"], rho2=pr["rho"][0],
                         rho3=pr["rho"][1], tau2=pr["tau"][0], tau3=pr["tau"][1],
                         body=pr["body"], faces=pr["faces"])


class _Study:
    """A served request as the executor admits it."""

    def __init__(self, shape, seed):
        rng = random.Random(seed)
        self.shape, self.n = shape, math.prod(shape)
        self.lattice = "D2Q9" if len(shape) == 2 else "D3Q19"
        self.theta_deg = rng.uniform(30.0, 150.0)
        sd, c2 = _request(shape, rng)
        c2 = (c2 + _noise(_gen(seed), c2.shape, torch.float64)) * (1 - _profile(sd, WIDTH3))
        self.solid_sd, self.c2 = sd.float().reshape(-1), c2.float().reshape(-1).contiguous()
        self.g12 = self.g23 = 2.5e-3
        self.alpha, self.alpha_s = 1.0, WIDTH3
        self.rho2 = self.rho3 = self.tau2 = self.tau3 = self.tau_g = 1.0
        self.body, self.faces = (0.0, 0.0, 0.0), None
        self.payload = self


def _sides(case):
    """Sides of a quantum's lattices: 2D from 64 to 512, 3D from 64 to 160."""
    flat = [64 + (448 * (2 * k + 1)) // (2 * case["flat"]) for k in range(case["flat"])]
    solid = [max(64, case["side"] * (3 - k) // 3) for k in range(case["solid"])]
    return flat, solid


def _studies(case, seed):
    flat, solid = _sides(case)
    shapes = [(s, s) for s in flat] + [(s, s, s) for s in solid]
    return [_Study(s, 1000 * seed + k) for k, s in enumerate(shapes)]


def _em_problem(case, seed):
    """A drop on a sinusoidal wall: parameters, solid, liquid, target volume."""
    rng = random.Random(seed)
    flat = case["nz"] == 1
    shape = (case["nx"], case["ny"]) if flat else (case["nx"], case["ny"], case["nz"])
    X = _coords(shape)
    base, amp = 16.0, 6.0
    k = 2 * math.pi / 32.0
    phase = rng.uniform(0, 2 * math.pi)
    slope = amp * k * torch.cos(k * X[0] + phase)
    sd = (base + amp * torch.sin(k * X[0] + phase) - X[-1]) / (1 + slope * slope).sqrt()
    c1 = _profile(sd.expand(shape[::-1]), 1.0)
    centre = [s / 2.0 for s in shape]
    centre[-1] = base + amp
    r = sum((X[a] - centre[a]) ** 2 for a in range(len(shape))).sqrt()
    radius = 0.235 * min(shape)
    c2 = 0.5 * (1 + torch.tanh((radius - r) / 2)) * (1 - c1)
    c2 = c2 + 0.1 * _noise(_gen(seed), c2.shape, torch.float64)
    c1, c2 = c1.float().reshape(-1).contiguous(), c2.float().reshape(-1).contiguous()
    V0 = 0.999 * float(c2.double().sum())
    return dict(lattice="D2Q9" if flat else "D3Q19", shape=shape, theta=rng.uniform(100.0, 130.0),
                g23=math.sqrt(8.0 / 9.0), g12=1.0, c1=c1, c2=c2, V0=V0, kcs=1e-2)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("energy", "lbfgs"):
        em = _em_problem(case, seed)
        p = P.make_params(em["lattice"], em["shape"], "f32", theta_deg=em["theta"], g23=em["g23"],
                          g12=em["g12"])
        return dict(case=case, em=em, fe=FreeEnergy(p), x=em["c2"].clone().requires_grad_(True))
    if kind == "served":
        ex = GpuExecutor("f32", angles=False)
        lats = [ex.admit(s) for s in _studies(case, seed)]
        return dict(case=case, ex=ex, lats=lats)
    pr = _problem(case, seed)
    if kind == "multi":
        kappa = P._lib.dsm_kappa(_params(pr))
        n = case["nfluid"]
        lat = P.MultiLattice(_params(pr), n, [kappa[0]] + [kappa[1]] * (n - 1) + [kappa[2]],
                             (1.0,) * n, (1.0,) * n)
        lat.set_solid_c1(pr["c1"])
        lat.set_fluids(pr["C"])
        return dict(case=case, lat=lat)
    lat = P.Lattice(_params(pr))
    if kind == "relax":
        return dict(case=case, lat=lat, pr=pr)
    if kind == "request":
        return dict(case=case, lat=lat, pr=pr)
    lat.set_solid_c1(pr["c1"])
    lat.set_fluid(pr["c2"])
    return dict(case=case, lat=lat)


# -------------------------------------------------------------------- pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "energy":
        em, x = state["em"], state["x"]
        x.grad = None
        E = Energy.apply(x, em["c1"], state["fe"], 2, None, 0.0, em["kcs"], em["V0"])
        E.backward()
        return {"E": E.detach(), "grad": x.grad}
    if kind == "lbfgs":
        em = state["em"]
        x, E, info = lbfgs(state["fe"], em["c2"], em["c1"], kcs=em["kcs"], V0=em["V0"], tol=0.0,
                           max_iter=case["iters"])
        return {"x": x, "E": E, "iterations": info["iterations"]}
    if kind == "served":
        state["ex"].advance([(lat, case["steps"]) for lat in state["lats"]])
        out = [lat.field("C2") for lat in state["lats"]]
        for lat in state["lats"]:   # each on its own stream: complete before use
            lat.stream.synchronize()
        return out
    lat = state["lat"]
    if kind == "relax":
        pr = state["pr"]
        lat.set_solid_c1(pr["c1"])
        lat.relax_solid(pr["mask"], case["steps"], pr["beta"], pr["omega"])
        return lat.field("C1")
    if kind == "request":
        lat.set_solid_distance(state["pr"]["sd"])
        lat.set_fluid(state["pr"]["c2"])
    lat.step(case["steps"])
    if kind == "multi":
        f, g = lat.populations()
        return {"f": f, "g": g}
    if kind in ("slab", "drop64"):
        f, g = lat.populations()
        return {"f": f, "g": g}
    return {"C2": lat.field("C2"), "pt": lat.field("pt")}


def _nodes(case):
    return case["nx"] * case["ny"] * case.get("nz", 1)


def work(case):
    """Bytes and operations a pass cannot do without.  Of a lattice's state a
    step reads and writes what fixes it: with every relaxation time 1 the
    hydrodynamic moments and the order parameter's (9 reals in 3D, 7 in 2D, 2
    more per further fluid), else the populations f beside u, mu and C."""
    kind = case["kind"]
    if kind == "energy":
        n = _nodes(case)
        return {"bytes": 16.0 * n, "flops": 200.0 * n}   # C1, C2 in; gradient out, scaled
    if kind == "lbfgs":
        n = _nodes(case)
        # per iteration the 20 stored vectors twice, 8 more and the energy's
        return {"bytes": case["iters"] * 4.0 * (40 + 8 + 3) * n, "flops": case["iters"] * 300.0 * n}
    if kind == "served":
        flat, solid = _sides(case)
        n2, n3 = sum(s ** 2 for s in flat), sum(s ** 3 for s in solid)
        return {"bytes": case["steps"] * (60.0 * n2 + 76.0 * n3),
                "flops": case["steps"] * (200.0 * n2 + 500.0 * n3)}
    n, k = _nodes(case), case["steps"]
    two_d = "nz" not in case
    q = 9 if two_d else 19
    reals = 7 if two_d else 9
    if kind == "multi":
        reals += 2 * (case["nfluid"] - 2)
    if kind in ("contrast", "plates", "channel"):
        reals = q + 5
    if kind == "plates":
        size = (q * 2.0 + 5 * 4.0) * 2 + 4.0
    else:
        size = (2 * reals + 1) * (8.0 if kind == "drop64" else 4.0)
    return {"bytes": k * n * size, "flops": k * n * (200.0 if two_d else 500.0)}


# ------------------------------------------------- the same pass in 64 bits
def _lattice(name):
    if name == "D2Q9":
        c = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    else:
        c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
             (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
             (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    return c, w


class _Exact:
    """Plain torch FP64 statement of the method for N fluids (N = 2: two), on
    arrays of shape (nz, ny, nx) or (ny, nx)."""

    def __init__(self, lattice, shape, kappa, rho, tau, body, faces, alpha_s, c1):
        self.c, self.w = _lattice(lattice)
        self.d, self.shape = len(shape), shape
        self.opp = [self.c.index(tuple(-v for v in ci)) for ci in self.c]
        self.kappa, self.rho, self.tau = kappa, rho, tau
        self.body, self.alpha_s = body, alpha_s
        self.face = [(0, 0)] * self.d
        for a in range(self.d):
            self.face[a] = tuple({"periodic": 0, "mirror": 1, "wall": 2}[f]
                                 for f in faces[2 * a:2 * a + 2])
        self.dims = tuple(reversed(shape))
        if c1 is not None:
            self.c1 = c1.double().reshape(self.dims)
            self.n1 = [self.at(self.c1, ci) for ci in self.c]
            self.solid = self.c1 >= 0.5
            self.lap1, self.g1 = self.lap(self.c1, self.n1), self.grad(self.n1)
            self.links = self._links()

    def at(self, v, off):
        """v at x + off; beyond a mirror or wall face the edge node."""
        for a, o in enumerate(off):
            if o == 0:
                continue
            dim, n = self.d - 1 - a, self.shape[a]
            r = torch.roll(v, -o, dim)
            if o > 0 and self.face[a][1]:
                r.narrow(dim, n - 1, 1).copy_(v.narrow(dim, n - 1, 1))
            if o < 0 and self.face[a][0]:
                r.narrow(dim, 0, 1).copy_(v.narrow(dim, 0, 1))
            v = r
        return v

    def lap(self, v, nb):
        s = torch.zeros_like(v)
        for w, m in zip(self.w[1:], nb[1:]):
            s += w * (m - v)
        return 6.0 * s

    def grad(self, nb):
        out = []
        for a in range(self.d):
            s = 0.0
            for ci, w, m in zip(self.c, self.w, nb):
                if ci[a]:
                    s = s + w * ci[a] * m
            out.append(3.0 * s)
        return out

    def _cross(self, j):
        """Where the link pulled in direction j crosses a face: (mask of wall
        crossings, list of (mask, direction read) of mirror crossings)."""
        zero = torch.zeros(self.dims, dtype=torch.bool, device=DEV)
        wall, per_axis = zero.clone(), []
        for a, o in enumerate(self.c[j]):
            side = self.face[a][0 if o > 0 else 1] if o else 0
            m = zero.clone()
            if side:
                m.narrow(self.d - 1 - a, 0 if o > 0 else self.shape[a] - 1, 1).fill_(True)
                if side == 2:
                    wall |= m
            per_axis.append(m)
        mirror = []
        if any(any(f) for f in self.face):
            for bits in range(1, 1 << self.d):
                m = ~wall
                ck = list(self.c[j])
                for a in range(self.d):
                    m = m & (per_axis[a] if bits >> a & 1 else ~per_axis[a])
                    if bits >> a & 1:
                        ck[a] = -ck[a]
                if bool(m.any()):
                    mirror.append((m, self.c.index(tuple(ck))))
        return wall, mirror

    def pull(self, f):
        """Populations streamed into every node, face rules included."""
        out = []
        for j, ci in enumerate(self.c):
            back = tuple(-v for v in ci)
            v = self.at(f[j], back)
            wall, mirror = self.crossings[j]
            for m, k in mirror:
                v = torch.where(m, self.at(f[k], back), v)
            if self.faced:
                v = torch.where(wall, f[self.opp[j]], v)
            out.append(v)
        return out

    @property
    def faced(self):
        return any(any(f) for f in self.face)

    def _links(self):
        """Interpolated bounce-back: the nodes of every link from the solid, the
        link fraction there, and whether the next node away is fluid."""
        self.crossings = [self._cross(j) for j in range(len(self.c))]
        links = []
        xs = 2.0 * self.alpha_s * torch.atanh(2.0 * self.c1.clamp(1e-9, 0.5) - 1.0)
        gn = sum(g * g for g in self.g1).sqrt()
        for j in range(1, len(self.c)):
            i = self.opp[j]
            hit = (~self.solid) & (self.n1[i] >= 0.5) & ~self.crossings[j][0]
            at = hit.reshape(-1).nonzero().reshape(-1)
            cl = math.sqrt(sum(v * v for v in self.c[i]))
            pick = [t.reshape(-1)[at] for t in (xs, gn, *self.g1)]
            nd = sum(g * v for g, v in zip(pick[2:], self.c[i])) / (pick[1] * cl)
            q = (pick[0] / nd).abs() / cl
            q = torch.where((pick[1] >= 1e-12) & (nd > 1e-6) & (q <= 1.0), q,
                            torch.full_like(q, 0.5))
            second = ((self.n1[j] < 0.5) & ~self.crossings[i][0]).reshape(-1)[at]
            links.append((j, i, at, q, second))
        return links

    def wells(self, c):
        return c * (1 - c) * (1 - 2 * c)

    def potentials(self, C):
        """mu_f of every free fluid, with what else the step needs of C."""
        nb = [[self.at(c, ci) for ci in self.c] for c in C]
        laps = [self.lap(c, m) for c, m in zip(C, nb)]
        last = 1.0 - self.c1 - sum(C)
        d = [self.kappa[1 + f] * (self.wells(c) - laps[f]) for f, c in enumerate(C)]
        dl = self.kappa[-1] * (self.wells(last) + self.lap1 + sum(laps))
        return [v - dl for v in d], nb, last

    def rho_of(self, C, c1):
        free = 1.0 - c1
        r = torch.full_like(c1, self.rho[-1])
        for f, c in enumerate(C):
            ph = torch.where(free > 1e-6, c / free.clamp(min=1e-6), torch.zeros_like(c))
            r += (self.rho[f] - self.rho[-1]) * ph.clamp(0.0, 1.0)
        return r

    def init(self, C):
        mu = self.potentials(C)[0]
        f = [torch.full(self.dims, w, dtype=torch.float64, device=DEV) for w in self.w]
        g = [self.geq(c, m, [torch.zeros_like(c)] * self.d) for c, m in zip(C, mu)]
        return f, g

    def s(self, i, u, uu):
        cu = sum(v * x for v, x in zip(self.c[i], u) if v)
        return 3.0 * cu + 4.5 * cu * cu - 1.5 * uu

    def geq(self, C, mu, u):
        uu = sum(x * x for x in u)
        out = [C - (1 - self.w[0]) * mu - self.w[0] * C * 1.5 * uu]
        for i in range(1, len(self.c)):
            out.append(self.w[i] * (mu + C * self.s(i, u, uu)))
        return out

    def moments(self, f, g):
        """Fields of the streamed state: C_f, mu_f, rho, tau, u, pt and the
        forces and streamed populations the collision needs."""
        C = [sum(self.pull(gf)) for gf in g]
        mu, nb, last = self.potentials(C)
        rho = self.rho_of(C, self.c1)
        contrast = any(r != self.rho[-1] for r in self.rho)
        gR = [torch.zeros_like(rho)] * self.d
        if contrast:
            gR = self.grad([self.rho_of([m[i] for m in nb], self.n1[i])
                            for i in range(len(self.c))])
        tau = torch.full_like(rho, self.tau[-1])
        big = last.clone()
        for k in range(len(C) - 1, -1, -1):
            more = C[k] > big
            tau, big = torch.where(more, torch.full_like(tau, self.tau[k]), tau), \
                torch.maximum(big, C[k])
        F = [self.body[a] * C[0] for a in range(self.d)]
        for m, n in zip(mu, nb):
            for a, gr in enumerate(self.grad(n)):
                F[a] = F[a] + m * gr
        del nb
        fs = self.pull(f)
        raw = list(fs)
        for j, i, at, q, second in self.links:
            fi, fz, fj = (t.reshape(-1)[at] for t in (f[i], raw[i], f[j]))
            v = torch.where(q < 0.5, torch.where(second, 2 * q * fi + (1 - 2 * q) * fz, fi),
                            fi / (2 * q) + (1 - 1 / (2 * q)) * fj)
            t = fs[j].clone()
            t.reshape(-1)[at] = v
            fs[j] = t
        u = []
        for a in range(self.d):
            m = sum(ci[a] * x for ci, x in zip(self.c, fs) if ci[a])
            u.append(torch.where(self.solid, torch.zeros_like(m), (m + 0.5 * F[a]) / rho))
        pt = sum(fs) + 0.5 * sum(x * y for x, y in zip(u, gR))
        pt = torch.where(self.solid, torch.ones_like(pt), pt)
        return C, mu, rho, tau, u, pt, F, gR, fs

    def step(self, f, g):
        C, mu, rho, tau, u, pt, F, gR, fs = self.moments(f, g)
        g = [self.geq(c, m, u) for c, m in zip(C, mu)]   # tau_g = 1
        uu = sum(x * x for x in u)
        ug = sum(x * y for x, y in zip(u, gR))
        kF = 1.0 - 0.5 / tau
        out = []
        for i, w in enumerate(self.w):
            s = self.s(i, u, uu)
            cF = sum(v * x for v, x in zip(self.c[i], F) if v)
            cg = sum(v * x for v, x in zip(self.c[i], gR) if v)
            v = fs[i] + (w * (pt + rho * s) - fs[i]) / tau + kF * w * ((cg - ug) * s + 3.0 * cF)
            out.append(torch.where(self.solid, torch.full_like(v, w), v))
        return out, g

    def relax(self, c1, mask, beta, omega, steps, k13):
        """Stage 1: the solid itself relaxed toward its region."""
        self.crossings = [self._cross(j) for j in range(len(self.c))]
        inside = mask.reshape(self.dims) != 0

        def mu_of(c):
            nb = [self.at(c, ci) for ci in self.c]
            mu = k13 * (self.wells(c) - self.lap(c, nb))
            leak = (inside & (c < 0.5)) | (~inside & (c > 0.5))
            mu = mu + torch.where(leak, 2 * beta * (c - 0.5), torch.zeros_like(c))
            return mu + 2 * omega * torch.where(c < 0, c, torch.where(
                c > 1, c - 1, torch.zeros_like(c))), self.grad(nb)

        c = c1.double().reshape(self.dims)
        f = [torch.full_like(c, w) for w in self.w]
        g = self.geq(c, mu_of(c)[0], [torch.zeros_like(c)] * self.d)
        for _ in range(steps):
            c = sum(self.pull(g))
            mu, gr = mu_of(c)
            fs = self.pull(f)
            u = [sum(ci[a] * x for ci, x in zip(self.c, fs) if ci[a]) + 0.5 * mu * gr[a]
                 for a in range(self.d)]
            pt, uu = sum(fs), sum(x * x for x in u)
            f = [w * (pt + self.s(i, u, uu) + 1.5 * mu * sum(
                v * x for v, x in zip(self.c[i], gr))) for i, w in enumerate(self.w)]
            g = self.geq(c, mu, u)
        return sum(self.pull(g))


def _kappa(theta, g12, g23):
    g13 = g12 + g23 * math.cos(math.radians(theta))
    return [3.0 * (g12 + g13 - g23), 3.0 * (g12 - g13 + g23), 3.0 * (-g12 + g13 + g23)]


def _exact_run(lattice, shape, kappa, rho, tau, body, faces, alpha_s, c1, C, steps):
    ex = _Exact(lattice, shape, kappa, rho, tau, body, faces, alpha_s, c1)
    f, g = ex.init([c.double().reshape(ex.dims) for c in C])
    for _ in range(steps):
        f, g = ex.step(f, g)
    return ex, f, g


def exact(case, seed):
    kind = case["kind"]
    if kind == "lbfgs":
        return None
    if kind == "energy":
        return _exact_energy(_em_problem(case, seed))
    if kind == "served":
        out = []
        for s in _studies(case, seed):
            body = (0.0,) * len(s.shape)
            ex, f, g = _exact_run(s.lattice, s.shape, _kappa(s.theta_deg, s.g12, s.g23),
                                  (1.0, 1.0), (1.0, 1.0), body, PERIODIC, s.alpha_s,
                                  _profile(s.solid_sd.double(), s.alpha_s), [s.c2],
                                  case["steps"])
            out.append(sum(ex.pull(g[0])).reshape(-1))
        return out
    pr = _problem(case, seed)
    kappa = _kappa(pr["theta"], pr["g12"], pr["g23"])
    if kind == "relax":
        ex = _Exact(pr["lattice"], pr["shape"], kappa, None, None, None, pr["faces"], None, None)
        return ex.relax(pr["c1"], pr["mask"], pr["beta"], pr["omega"], case["steps"],
                        kappa[0] + kappa[2]).reshape(-1)
    c1, C, rho, tau = pr["c1"], [pr["c2"]], pr["rho"], pr["tau"]
    if kind == "request":
        c1 = _profile(pr["sd"].double(), pr["alpha_s"])
    if kind == "multi":
        n = case["nfluid"]
        C, rho, tau = list(pr["C"]), (1.0,) * n, (1.0,) * n
        kappa = [kappa[0]] + [kappa[1]] * (n - 1) + [kappa[2]]
    body = pr["body"][:len(pr["shape"])]
    ex, f, g = _exact_run(pr["lattice"], pr["shape"], kappa, rho, tau, body, pr["faces"],
                          pr["alpha_s"], c1, C, case["steps"])
    if kind in ("slab", "drop64", "multi"):
        return {"f": torch.stack(f).reshape(-1),
                "g": torch.stack([x for y in g for x in y]).reshape(-1)}
    C, _, _, _, _, pt = ex.moments(f, g)[:6]
    return {"C2": C[0].reshape(-1), "pt": pt.reshape(-1)}


def _exact_energy(em):
    kappa = _kappa(em["theta"], em["g12"], em["g23"])
    ex = _Exact(em["lattice"], em["shape"], kappa, None, None, None, PERIODIC, None, None)
    c1, c2 = (em[k].double().reshape(ex.dims) for k in ("c1", "c2"))
    fields = [c1, c2, 1.0 - c1 - c2]
    E, d = 0.0, []
    for k, c in zip(kappa, fields):
        nb = [ex.at(c, ci) for ci in ex.c]
        pair = sum(w * (m - c) ** 2 for w, m in zip(ex.w, nb))
        E = E + (0.5 * k * (c * (1 - c)) ** 2 + 1.5 * k * pair).sum()
        d.append(k * (ex.wells(c) - ex.lap(c, nb)))
    V = c2.sum()
    E = E + 0.5 * em["kcs"] * (V - em["V0"]) ** 2
    return {"E": E, "grad": (d[1] - d[2] + em["kcs"] * (V - em["V0"])).reshape(-1)}
