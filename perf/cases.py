"""Timed cases: what users of this library run, through its public entry points.

A pass of a single simulation is one output interval: so many time steps, then
the density, velocity and node positions read into the host buffers that the
program keeps, and the observables (or the deformation index in shear).  A
pass of a batch is the same for all its slots.  A campaign is a whole call of
serve.run_batched: admission, every step, results.

Fields and observables come back in the compute precision of the storage
form: FP64 for FP64 storage, FP32 for FP32 and binary16 storage.

exact() advances the same problems with the paper's formulas written out in
FP64 torch operations; it takes only the initial shapes from the package.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2604_17463_gb300 import iblb, serve
from paper_2604_17463_gb300 import workloads as W

STORAGE = {"fp64": iblb.FP64, "fp32": iblb.FP32_DEV, "fp16": iblb.FP16_DEV}
ELT = {"fp64": 8, "fp32": 4, "fp16": 2}


# ------------------------------------------------------------------ the cases
def case(name, shape, storage, steps, *, nx=0, ny=0, nz=1, count=1, autotune=False, ordered=False,
         elastic=False, lam=1.0):
    return {"name": name, "shape": shape, "storage": storage, "steps": steps, "nx": nx, "ny": ny,
            "nz": nz, "count": count, "autotune": autotune, "ordered": ordered, "elastic": elastic,
            "lam": lam}


def listed():
    return [
        # the small FP64 drop of the smoke check and the tests, watched closely
        case("ring_128x64_fp64", "drop2d", "fp64", 50, nx=128, ny=64),
        # the 2D spreading study: one parameter point between two outputs
        case("spread_2048x512_fp32", "spread2d", "fp32", 500, nx=2048, ny=512),
        # the largest member of the batched workload on its own, binary16
        case("ring_1024x256_fp16", "drop2d", "fp16", 500, nx=1024, ny=256),
        # the 3D benchmark drop as the README runs it, and in binary16
        case("drop_256x256x128_fp32", "drop3d", "fp32", 200, nx=256, ny=256, nz=128, autotune=True),
        case("drop_256x256x128_fp16", "drop3d", "fp16", 200, nx=256, ny=256, nz=128, autotune=True),
        # a served 3D request of odd extent run alone, with default settings
        case("drop_101x101x77_fp32", "drop3d", "fp32", 300, nx=101, ny=101, nz=77),
        # the paper-scale spreading cap (118 580 triangles)
        case("cap_250x250x150_fp32", "cap3d", "fp32", 100, nx=250, ny=250, nz=150, autotune=True),
        # the drop in shear of the paper, with a viscosity ratio
        case("shear_160x128x242_fp32", "shear3d", "fp32", 100, nx=160, ny=128, nz=242, lam=0.5),
        # a bitwise reproducible FP64 run of a capsule
        case("capsule_96x96x72_fp64", "drop3d", "fp64", 50, nx=96, ny=96, nz=72, ordered=True,
             elastic=True),
        # a resident batch of uneven 2D drops, binary16 as the serving mode uses it
        case("batch_64_drops_fp16", "batch2d", "fp16", 1000, count=64),
        # a resident batch of 3D requests of the serving mix
        case("batch_8_drops3d_fp32", "batch3d", "fp32", 300, count=8),
        # a parameter campaign of 2D drops as one call
        case("campaign_48_drops_fp32", "campaign2d", "fp32", 2000, count=48),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: extents over their logarithm, mostly odd
    ones, every storage form and option."""
    shape = rng.choice(["drop2d", "drop2d", "spread2d", "drop3d", "drop3d", "shear3d", "batch2d",
                        "batch3d", "campaign2d"])
    storage = rng.choice(["fp32", "fp32", "fp16", "fp64"])
    autotune = rng.random() < 0.3
    ordered = rng.random() < 0.15
    elastic = rng.random() < 0.15
    kw = {"autotune": autotune, "ordered": ordered, "elastic": elastic}
    if shape == "drop2d":
        nx = _log_int(rng, 64, 2048)
        kw.update(nx=nx, ny=max(12, int(nx * rng.uniform(0.25, 0.5))))
        steps = _log_int(rng, 20, 500)
    elif shape == "spread2d":
        d = rng.choice([1, 2, 4])
        kw.update(nx=2048 // d, ny=512 // d)
        steps = _log_int(rng, 50, 500)
    elif shape == "drop3d":
        nx = _log_int(rng, 48, 224)
        kw.update(nx=nx, ny=max(32, int(nx * rng.uniform(0.8, 1.0))), nz=max(32, int(nx * rng.uniform(0.5, 0.7))))
        steps = _log_int(rng, 20, 100)
    elif shape == "shear3d":
        nx = _log_int(rng, 48, 160)
        kw.update(nx=nx, ny=max(40, int(0.8 * nx)), nz=max(42, int(1.5 * nx)), lam=rng.choice([0.5, 1.0, 2.0]))
        kw["elastic"] = False
        steps = _log_int(rng, 20, 100)
    elif shape == "batch2d":
        kw.update(count=_log_int(rng, 8, 96), elastic=False, autotune=False)
        steps = _log_int(rng, 100, 800)
    elif shape == "batch3d":
        kw.update(count=_log_int(rng, 2, 8), elastic=False, autotune=False)
        steps = _log_int(rng, 50, 250)
    else:
        kw.update(count=_log_int(rng, 4, 48), elastic=False, autotune=False)
        steps = _log_int(rng, 200, 2000)
    if storage == "fp64" and shape in ("batch2d", "batch3d", "campaign2d", "drop3d", "shear3d", "spread2d"):
        steps = max(10, steps // 10)
    c = case("", shape, storage, steps, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ the problems
@functools.lru_cache(maxsize=None)
def _level(radius):
    return W.icosphere_level_for(radius)


@functools.lru_cache(maxsize=None)
def _unit_sphere(level):
    return W.icosphere(level, 1.0, (0.0, 0.0, 0.0))


@functools.lru_cache(maxsize=None)
def _cap():
    return W.spread3d_cap(0.8).work


def _problem(lattice, dims, nodes, faces, rng, *, theta, tau, sigma=1e-3, xi, wetting=True, steps=0,
             tau_out=0.0, gs=0.0, uw=0.0, u0=None):
    return {"lattice": lattice, "dims": dims, "nodes": nodes, "faces": faces, "theta": theta,
            "tau": tau, "sigma": sigma, "xi": xi, "wetting": wetting, "steps": steps,
            "tau_out": tau_out, "gs": gs, "uw": uw, "u0": u0}


def _ring(nx, ny, rng, steps=0, gs=0.0):
    """A 2D drop at its film distance from the wall, its centre anywhere between
    lattice points."""
    n = max(16, int(round(10 * ny / 3.0)))
    R = ny / 3.0 * rng.uniform(0.95, 1.0)
    xi = max(0.05 * R, 1.0)
    nodes = W.circle(n, R, (nx / 2.0 + rng.uniform(-0.5, 0.5), W.WALL_PLANE + R + xi))
    return _problem(9, (nx, ny, 1), nodes, None, rng, theta=rng.uniform(45.0, 105.0),
                    tau=rng.uniform(0.7, 1.2), xi=xi, steps=steps, gs=gs)


def _ball(nx, ny, nz, rng, gs=0.0):
    """A 3D drop, mesh edges of at most about 1.5 lattice units."""
    R0 = min(nz / 3.0, 0.4 * min(nx, ny), 40.0)
    unit, faces = _unit_sphere(_level(R0))
    R = R0 * rng.uniform(0.97, 1.0)
    xi = max(0.05 * R, 1.0)
    nodes = unit * R + np.array([nx / 2.0 + rng.uniform(-0.5, 0.5), ny / 2.0 + rng.uniform(-0.5, 0.5),
                                 W.WALL_PLANE + R + xi])
    return _problem(19, (nx, ny, nz), nodes, faces, rng, theta=rng.uniform(45.0, 105.0),
                    tau=rng.uniform(0.7, 1.1), xi=xi, gs=gs)


def _problems(c, seed):
    rng = np.random.default_rng(seed)
    gs = 1e-3 if c["elastic"] else 0.0
    if c["shape"] == "drop2d":
        return [_ring(c["nx"], c["ny"], rng, gs=gs)]
    if c["shape"] == "spread2d":
        wl = W.spreading_2d_2048x512(downscale=2048 // c["nx"])
        nodes = wl.nodes + np.array([rng.uniform(-0.5, 0.5), rng.uniform(0.0, 0.3)])
        return [_problem(9, (wl.nx, wl.ny, 1), nodes, None, rng, theta=rng.uniform(45.0, 105.0),
                         tau=rng.uniform(0.7, 1.1), xi=wl.xi, gs=gs)]
    if c["shape"] == "drop3d":
        return [_ball(c["nx"], c["ny"], c["nz"], rng, gs=gs)]
    if c["shape"] == "cap3d":
        wl = _cap()
        nodes = wl.nodes + np.array([rng.uniform(-0.5, 0.5), rng.uniform(-0.5, 0.5), rng.uniform(0.0, 0.3)])
        return [_problem(19, (wl.nx, wl.ny, wl.nz), nodes, wl.faces, rng, theta=rng.uniform(55.0, 75.0),
                         tau=rng.uniform(0.7, 1.1), xi=wl.xi)]
    if c["shape"] == "shear3d":
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        R = 19.0 * min(1.0, nx / 160.0) * rng.uniform(0.95, 1.0)
        unit, faces = _unit_sphere(5 if R > 12 else 4)
        nodes = unit * R + np.array([nx / 2.0 + rng.uniform(0.1, 0.4), ny / 2.0 - rng.uniform(0.1, 0.4),
                                     nz / 2.0 - 0.5 + rng.uniform(0.05, 0.2)])
        tau = 1.0
        tau_out = 0.5 + (tau - 0.5) / c["lam"]
        uw = rng.uniform(0.01, 0.02)
        H = nz - 2.0
        prof = 2.0 * uw / H * (np.arange(nz) - (nz - 1) / 2.0)
        prof[0] = prof[-1] = 0.0
        u0 = np.zeros((3, nz, ny, nx))
        u0[0] = prof[:, None, None]
        return [_problem(19, (nx, ny, nz), nodes, faces, rng, theta=90.0, tau=tau, sigma=5e-3, xi=0.05 * R,
                         wetting=False, tau_out=tau_out, uw=uw, u0=u0)]
    sizes = np.random.default_rng(7)  # the members' sizes belong to the case, their drops to the seed
    out = []
    for _ in range(c["count"]):
        if c["shape"] == "batch3d":
            s = sizes.uniform(0.0, 1.0)
            nx, nz = int(round(64 + s * (192 - 64))), int(round(64 + s * (96 - 64)))
            out.append(_ball(nx, nx, nz, rng))
        else:
            w = int(round(math.exp(sizes.uniform(math.log(64), math.log(1024)))))
            steps = int(sizes.integers(c["steps"] // 4, c["steps"] + 1))
            out.append(_ring(w, max(w // 4, 12), rng, steps=steps))
    return out


def _config(p, storage, ordered):
    nx, ny, nz = p["dims"]
    return dict(tau=p["tau"], walls=True, wetting=p["wetting"], sigma=p["sigma"], xi=p["xi"],
                theta_eq_deg=p["theta"], storage=storage, tau_out=p["tau_out"],
                wall_u_lo=(-p["uw"], 0.0, 0.0), wall_u_hi=(p["uw"], 0.0, 0.0),
                deterministic_spread=ordered, shear_modulus=p["gs"])


def _workload(p):
    nx, ny, nz = p["dims"]
    return W.Workload("drop", p["lattice"], nx, ny, nz, p["tau"], p["sigma"], p["xi"], p["theta"], 9, 3,
                      p["steps"], p["nodes"], p["faces"])


def prepare(c, seed):
    probs = _problems(c, seed)
    storage = STORAGE[c["storage"]]
    st = {"case": c, "dtype": torch.float64 if c["storage"] == "fp64" else torch.float32}
    if c["shape"] == "campaign2d":
        st["work"] = [_workload(p) for p in probs]
        return st
    if c["count"] == 1 and not c["shape"].startswith("batch"):
        p = probs[0]
        nx, ny, nz = p["dims"]
        sim = iblb.Simulation(p["lattice"], nx, ny, nz, **_config(p, storage, c["ordered"]))
        sim.set_interface(p["nodes"], p["faces"])
        if p["u0"] is not None:
            sim.set_equilibrium(p["u0"])
        if c["autotune"]:
            sim.autotune()
        st["sim"] = sim
        # page-locked result buffers, as a program that reads often keeps
        st["rho"] = torch.zeros(sim.shape, dtype=torch.float64).pin_memory()
        st["u"] = torch.zeros((sim.dim,) + sim.shape, dtype=torch.float64).pin_memory()
        st["q"] = torch.zeros((sim.N, sim.dim), dtype=torch.float64).pin_memory()
        return st
    lattice = probs[0]["lattice"]
    cfgs = []
    for p in probs:
        nx, ny, nz = p["dims"]
        cfgs.append(iblb.make_config(lattice, nx, ny, nz, **_config(p, storage, c["ordered"])))
    need = sum(iblb.Batch.footprint(f, len(p["nodes"]), 0 if p["faces"] is None else len(p["faces"]))
               for f, p in zip(cfgs, probs))
    b = iblb.Batch(lattice, storage, int(need * 1.02) + (1 << 20), max_slots=len(probs))
    st["batch"] = b
    st["slots"] = [b.admit(f, p["nodes"], p["faces"], 1 << 40) for f, p in zip(cfgs, probs)]
    return st


def _obs_row(o):
    return [o["mass"], o["volume"], o["height"], o["theta_deg"], o["r_cl"], o["film"], o["d_min"],
            *o["centre"], o["radius"]]


def run(st):
    c, dt = st["case"], st["dtype"]
    if "work" in st:
        r = serve.run_batched(st["work"], STORAGE[c["storage"]], 4 << 30)
        return torch.tensor([_obs_row(o) for o in r["obs"]], dtype=torch.float64).to(dt)
    if "sim" in st:
        sim = st["sim"]
        sim.step(c["steps"])
        iblb.iblb_read_fields(sim.h, st["rho"].numpy(), st["u"].numpy(), st["q"].numpy())
        out = {"rho": st["rho"].to(dt), "u": st["u"].to(dt), "q": st["q"].to(dt)}
        if c["shape"] == "shear3d":
            d = sim.deformation()
            out["shear"] = torch.tensor([d["D"], d["r1"], d["r3"], d["angle_deg"], d["volume"]],
                                        dtype=torch.float64).to(dt)
        else:
            out["obs"] = torch.tensor(_obs_row(sim.observables()), dtype=torch.float64).to(dt)
        return out
    b = st["batch"]
    b.run(c["steps"])
    got = [b.fields(s) for s in st["slots"]]
    return {k: torch.cat([torch.from_numpy(f[i]).reshape(-1) for f in got]).to(dt)
            for i, k in enumerate(("rho", "u", "q"))}


def work(c):
    """Populations read once and written once per fluid cell and step, and the
    results written once; the interface's bytes are below a percent of that."""
    elt = ELT[c["storage"]]
    by = fl = 0.0
    for p in _problems(c, 0):
        nx, ny, nz = p["dims"]
        q, dim = p["lattice"], 2 if p["lattice"] == 9 else 3
        fluid = nx * (ny - 2) if dim == 2 else nx * ny * (nz - 2)
        steps = p["steps"] if c["shape"] == "campaign2d" else c["steps"]
        by += steps * 2.0 * q * elt * fluid
        fl += steps * fluid * (120.0 if dim == 2 else 270.0)
        if c["shape"] != "campaign2d":
            by += 8.0 * (1 + dim) * nx * ny * nz
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ 64-bit reference
VEL = {
    9: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)],
    19: [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
         (1, 1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, -1), (0, 1, 1), (0, -1, -1),
         (1, -1, 0), (-1, 1, 0), (1, 0, -1), (-1, 0, 1), (0, 1, -1), (0, -1, 1)],
}
WEIGHT = {9: {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}, 19: {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}}


def _delta(r):
    a = r.abs()
    near = (3 - 2 * a + torch.sqrt((1 + 4 * a - 4 * a * a).clamp_min(0))) / 8
    far = (5 - 2 * a - torch.sqrt((-7 + 12 * a - 4 * a * a).clamp_min(0))) / 8
    return torch.where(a <= 1, near, torch.where(a <= 2, far, torch.zeros_like(a)))


class _Exact:
    """Any number of independent problems of one lattice as one list of cells
    and one list of nodes."""

    def __init__(self, probs):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.dev, self.Q = dev, probs[0]["lattice"]
        self.dim = 2 if self.Q == 9 else 3
        self.vel = VEL[self.Q]
        self.opp = [self.vel.index(tuple(-k for k in v)) for v in self.vel]
        self.w = [WEIGHT[self.Q][sum(k * k for k in v)] for v in self.vel]
        f8 = dict(dtype=torch.float64, device=dev)
        self.ncell = sum(math.prod(p["dims"]) for p in probs)
        N, wax = self.ncell, self.dim - 1
        self.src = torch.empty((self.Q, N), dtype=torch.int64, device=dev)
        self.gain = torch.zeros((self.Q, N), **f8) if any(p["uw"] for p in probs) else None
        self.fluid = torch.empty(N, dtype=torch.bool, device=dev)
        self.omega = torch.empty(N, **f8)
        self.g = torch.zeros((self.Q, N), **f8)
        self.spans, q, per_node, base, nb = [], [], [], 0, 0
        prev, nxt, faces = [], [], []
        for p in probs:
            nx, ny, nz = p["dims"]
            n = nx * ny * nz
            cells = torch.arange(n, device=dev)
            xyz = [cells % nx, (cells // nx) % ny, cells // (nx * ny)]
            L = p["dims"][wax]
            a = xyz[wax]
            fl = (a > 0) & (a < L - 1)
            self.fluid[base:base + n] = fl
            self.omega[base:base + n] = 1.0 / p["tau"]
            for i, v in enumerate(self.vel):
                s = [(xyz[k] - v[k]) % p["dims"][k] for k in range(3)]
                sa = a - v[wax]
                bounce = fl & ((sa <= 0) | (sa >= L - 1))
                at = i * N + base + s[0] + nx * (s[1] + ny * s[2])
                self.src[i, base:base + n] = torch.where(bounce, self.opp[i] * N + base + cells, at)
                if p["uw"]:
                    side = (1.0 - 2.0 * (sa <= 0).double()) * bounce
                    self.gain[i, base:base + n] = 6 * self.w[i] * v[0] * p["uw"] * side
            if p["u0"] is not None:
                u = torch.tensor(p["u0"].reshape(self.dim, n), **f8)
                uu = (u * u).sum(0)
                for i, v in enumerate(self.vel):
                    cu = sum(v[k] * u[k] for k in range(self.dim))
                    self.g[i, base:base + n] = self.w[i] * (3 * cu + 4.5 * cu * cu - 1.5 * uu)
            m = len(p["nodes"])
            A = p["sigma"] * 16.0 / (6.0 * p["xi"]) * (1 + math.cos(math.radians(p["theta"]))) if p["wetting"] else 0.0
            per_node.append(torch.tensor([[base, nx, ny, nz, p["sigma"], p["xi"], A, p["gs"]]], **f8).expand(m, 8))
            q.append(torch.tensor(p["nodes"], **f8))
            if self.dim == 2:
                j = torch.arange(m, device=dev)
                prev.append(nb + (j - 1) % m)
                nxt.append(nb + (j + 1) % m)
            else:
                faces.append(nb + torch.tensor(p["faces"], dtype=torch.int64, device=dev))
            self.spans.append((base, n, nb, m))
            base += n
            nb += m
        self.q = torch.cat(q)
        par = torch.cat(per_node)
        self.base, self.ext = par[:, 0].long(), par[:, 1:4].long()
        self.sigma, self.xi, self.A, self.gs = par[:, 4], par[:, 5], par[:, 6], par[:, 7]
        if self.dim == 2:
            self.prev, self.next = torch.cat(prev), torch.cat(nxt)
        else:
            self.tri = torch.cat(faces)
        self.elastic = bool((self.gs != 0).any())
        if self.elastic:
            self.ref = self._reference()
        # a viscosity ratio is run one problem at a time
        p = probs[0]
        self.tau_out = p["tau_out"] if len(probs) == 1 and p["tau_out"] not in (0.0, p["tau"]) else 0.0
        self.tau, self.dims = p["tau"], p["dims"]

    # interface
    def _reference(self):
        if self.dim == 2:
            return (self.q[self.next] - self.q).norm(dim=1)
        P = self.q[self.tri]
        e1, e2 = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]
        x = e1 / e1.norm(dim=1, keepdim=True)
        n = torch.linalg.cross(e1, e2)
        y = torch.linalg.cross(n / n.norm(dim=1, keepdim=True), x)
        E = torch.stack([torch.stack([(e1 * x).sum(1), (e2 * x).sum(1)], 1),
                         torch.stack([(e1 * y).sum(1), (e2 * y).sum(1)], 1)], 1)
        return torch.linalg.inv(E), 0.5 * n.norm(dim=1)

    def _energy(self, q):
        """Surface energy plus Skalak's strain energy (C = 0)."""
        if self.dim == 2:
            ln = (q[self.next] - q).norm(dim=1)
            e = (self.sigma * ln).sum()
            if self.elastic:
                I = (ln / self.ref) ** 2 - 1
                e = e + (self.ref * self.gs / 4 * I * I).sum()
            return e
        P = q[self.tri]
        e1, e2 = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]
        own = self.tri[:, 0]
        e = (self.sigma[own] * 0.5 * torch.linalg.cross(e1, e2).norm(dim=1)).sum()
        if self.elastic:
            M, A0 = self.ref
            D = torch.stack([e1, e2], 2) @ M
            C = D.transpose(1, 2) @ D
            I1 = C[:, 0, 0] + C[:, 1, 1] - 2
            I2 = C[:, 0, 0] * C[:, 1, 1] - C[:, 0, 1] * C[:, 1, 0] - 1
            e = e + (A0 * self.gs[own] / 4 * (I1 * I1 + 2 * I1 - 2 * I2)).sum()
        return e

    def forces(self):
        q = self.q.detach().requires_grad_(True)
        phi = -torch.autograd.grad(self._energy(q), q)[0]
        q = self.q
        if self.dim == 2:
            s0, s1 = q - q[self.prev], q[self.next] - q
            l0, l1 = s0.norm(dim=1, keepdim=True), s1.norm(dim=1, keepdim=True)
            t = s0 / l0 + s1 / l1
            n = torch.stack([t[:, 1], -t[:, 0]], 1)
            chi, share = (l0 + l1)[:, 0], 0.5
        else:
            P = q[self.tri]
            c = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
            twice = c.norm(dim=1)
            n, chi = torch.zeros_like(q), torch.zeros_like(q[:, 0])
            for k in range(3):
                n.index_add_(0, self.tri[:, k], c / twice[:, None])
                chi.index_add_(0, self.tri[:, k], 0.5 * twice)
            share = 1 / 3
        n = n / n.norm(dim=1, keepdim=True)
        s = self.xi / (q[:, -1] - 0.5)
        pi = torch.where(self.A != 0, self.A * (s ** 9 - s ** 3), torch.zeros_like(s))
        return phi - share * (chi * pi)[:, None] * n

    def stencil(self):
        """Cells and weights of every node's 4^dim points; no weight on solid cells."""
        fl = torch.floor(self.q).long()
        o = torch.arange(-1, 3, device=self.dev)
        idx, wt = self.base[:, None], torch.ones_like(self.q[:, :1])
        stride = torch.ones_like(self.base)
        for k in range(self.dim):
            at = fl[:, k:k + 1] + o
            w = _delta(self.q[:, k:k + 1] - at)
            L = self.ext[:, k:k + 1]
            if k == self.dim - 1:
                w = torch.where((at > 0) & (at < L - 1), w, torch.zeros_like(w))
                at = torch.minimum(at.clamp_min(0), L - 1)
            else:
                at = at % L
            idx = (idx[:, :, None] + (at * stride[:, None])[:, None, :]).flatten(1)
            wt = (wt[:, :, None] * w[:, None, :]).flatten(1)
            stride = stride * self.ext[:, k]
        return idx, wt

    def classify(self):
        """Relaxation rate of every cell: an odd number of crossings of the
        interface below it along the wall axis is inside (3D, one problem)."""
        nx, ny, nz = self.dims
        P = self.q[self.tri]
        lo = torch.ceil(P[:, :, :2].amin(1))
        span = int((P[:, :, :2].amax(1) - lo).max().clamp_min(0)) + 1
        flip = torch.zeros((nz + 1) * ny * nx, dtype=torch.int64, device=self.dev)

        def edge(a, b, X, Y):
            return (b[:, 0] - a[:, 0]) * (Y - a[:, 1]) - (b[:, 1] - a[:, 1]) * (X - a[:, 0])

        for dx in range(span):
            for dy in range(span):
                X, Y = lo[:, 0] + dx, lo[:, 1] + dy
                w = [edge(P[:, (k + 1) % 3], P[:, (k + 2) % 3], X, Y) for k in range(3)]
                total = w[0] + w[1] + w[2]
                hit = (total != 0) & ((torch.stack(w) * torch.sign(total)) > 0).all(0)
                z = sum(w[k] * P[:, k, 2] for k in range(3)) / total
                first = (torch.floor(z[hit]).long() + 1).clamp(0, nz)
                at = X[hit].long() % nx + nx * (Y[hit].long() % ny + ny * first)
                flip.index_add_(0, at, torch.ones_like(at))
        inside = (flip.view(nz + 1, -1)[:nz].cumsum(0) % 2).reshape(-1).double()
        return inside * (1.0 / self.tau) + (1.0 - inside) * (1.0 / self.tau_out)

    def step(self):
        N, D = self.ncell, self.dim
        idx, wt = self.stencil()
        phi = self.forces()
        F = torch.zeros((D, N), dtype=torch.float64, device=self.dev)
        for k in range(D):
            F[k].index_add_(0, idx.reshape(-1), (phi[:, k:k + 1] * wt).reshape(-1))
        om = self.classify() if self.tau_out else self.omega
        g = torch.take(self.g, self.src)
        if self.gain is not None:
            g += self.gain
        rho = 1 + g.sum(0)
        u = torch.zeros_like(F)
        for i, v in enumerate(self.vel):
            for k in range(D):
                if v[k]:
                    u[k] += v[k] * g[i]
        u = (u + 0.5 * F) / rho
        uu, uF = (u * u).sum(0), (u * F).sum(0)
        for i, v in enumerate(self.vel):
            cu = sum(v[k] * u[k] for k in range(D) if v[k]) if i else 0.0
            cF = sum(v[k] * F[k] for k in range(D) if v[k]) if i else 0.0
            eq = self.w[i] * (rho - 1 + rho * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
            g[i] += om * (eq - g[i]) + (1 - 0.5 * om) * self.w[i] * (3 * (cF - uF) + 9 * cu * cF)
        self.g = g
        self.rho = torch.where(self.fluid, rho, torch.zeros_like(rho))
        self.u = torch.where(self.fluid, u, torch.zeros_like(u))
        self.q = self.q + torch.stack([(self.u[k][idx] * wt).sum(1) for k in range(D)], 1)

    # results
    def observables(self, k):
        base, n, nb, m = self.spans[k]
        q, D = self.q[nb:nb + m], self.dim
        xi = float(self.xi[nb])
        mass = float(self.rho[base:base + n].sum())
        if D == 2:
            r = torch.roll(q, -1, 0)
            vol = 0.5 * float((q[:, 0] * r[:, 1] - r[:, 0] * q[:, 1]).sum())
        else:
            P = q[self.tri]
            vol = float((P[:, 0] * torch.linalg.cross(P[:, 1], P[:, 2])).sum()) / 6
        z = q[:, -1]
        d_min = float(z.min()) - 0.5
        fit = q[z - 0.5 > 3 * xi]
        mean = fit.mean(0)
        v = fit - mean
        A = torch.cat([v, torch.ones_like(v[:, :1])], 1)
        s = torch.linalg.solve(A.T @ A, -(A.T @ (v * v).sum(1)))
        cen = -0.5 * s[:D]
        R = math.sqrt(float((cen * cen).sum() - s[D]))
        cen = cen + mean
        dz = d_min + 0.5 - float(cen[-1])
        theta = math.degrees(math.acos(min(1.0, max(-1.0, dz / R))))
        r_cl = math.sqrt(max(0.0, R * R - dz * dz))
        off = (q[:, :D - 1] - cen[:D - 1]).norm(dim=1)
        low = (off < 0.5 * r_cl) & (z - 0.5 <= 3 * xi)
        film = float((z[low] - 0.5).mean()) if bool(low.any()) else math.nan
        c3 = [float(cen[k]) if k < D else 0.0 for k in range(3)]
        return [mass, vol, float(z.max() - z.min()), theta, r_cl, film, d_min, *c3, R]

    def deformation(self):
        P = self.q[self.tri]
        P = P - self.q.mean(0)
        vol = (P[:, 0] * torch.linalg.cross(P[:, 1], P[:, 2])).sum(1) / 6
        s = P.sum(1)
        V = vol.sum()
        first = (vol[:, None] * s / 4).sum(0) / V
        second = (vol[:, None, None] / 20 * (torch.einsum("fvi,fvj->fij", P, P) + s[:, :, None] * s[:, None, :])).sum(0)
        S = second - V * first[:, None] * first[None, :]
        mean, half = 0.5 * float(S[0, 0] + S[2, 2]), 0.5 * float(S[0, 0] - S[2, 2])
        rad = math.hypot(half, float(S[0, 2]))
        r1, r3 = (math.sqrt(5 * (mean + t) / float(V)) for t in (rad, -rad))
        angle = math.degrees(0.5 * math.atan2(2 * float(S[0, 2]), 2 * half))
        return [(r1 - r3) / (r1 + r3), r1, r3, angle, float(V)]


def exact(c, seed):
    probs = _problems(c, seed)
    e = _Exact(probs)
    if c["shape"] == "campaign2d":
        rows = [None] * len(probs)
        for t in range(1, max(p["steps"] for p in probs) + 1):
            e.step()
            for k, p in enumerate(probs):
                if p["steps"] == t:
                    rows[k] = e.observables(k)
        return torch.tensor(rows, dtype=torch.float64)
    for _ in range(c["steps"]):
        e.step()
    if c["count"] == 1 and not c["shape"].startswith("batch"):
        nx, ny, nz = probs[0]["dims"]
        out = {"rho": e.rho.view(nz, ny, nx), "u": e.u.view(e.dim, nz, ny, nx), "q": e.q}
        if c["shape"] == "shear3d":
            out["shear"] = torch.tensor(e.deformation(), dtype=torch.float64)
        else:
            out["obs"] = torch.tensor(e.observables(0), dtype=torch.float64)
        return out
    return {"rho": e.rho, "u": torch.cat([e.u[:, b:b + n].reshape(-1) for b, n, _, _ in e.spans]), "q": e.q.reshape(-1)}
