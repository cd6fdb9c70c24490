"""The work that users of the library have it do, as measurable cases.

A case is one pass of a program that keeps its lattices (plan, weights and buffers) between
passes: it advances a state by some steps and reads it back ("run"), advances a batch of lattices
together ("ensemble"), or does one iteration of a flux fit, forward and reverse ("fit").  Sizes
and physics are those of the workloads in ``paper_2412_14859_gb300.inputs`` (and of the benchmark
geometries of the paper that the tests run), with drawn ones around them.

  listed()              the cases
  draw(rng)             one more case of the same ranges
  prepare(case, seed)   what the program has in hand before the call
  run(state)            one pass through the public entry points
  work(case)            bytes and operations a pass cannot do without
  exact(case, seed)     the pass's outputs in 64 bits, plain torch
"""
from __future__ import annotations

import math

import torch

from paper_2412_14859_gb300 import inputs
from paper_2412_14859_gb300.adjoint import volume_history
from paper_2412_14859_gb300.binding import Ensemble, Sim

HEATED_EVERY = 10   # steps between refreshes of a heated-substrate flux
FIT_COEFFICIENTS = 16


# ------------------------------------------------------------------ the cases ---------------

def _run(name, q, nx, ny, nz, storage, steps, geometry="drop", walls=False, rule="band",
         gamma=1.0, flux="scalar"):
    return {"name": name, "kind": "run", "q": q, "nx": nx, "ny": ny, "nz": nz, "storage": storage,
            "steps": steps, "geometry": geometry, "walls": walls, "rule": rule, "gamma": gamma,
            "flux": flux}


def listed():
    return [
        # the smallest lattice in use: the FP64 reference slab, a few steps between looks at its
        # fields; launches and one kernel's latency are all there is
        _run("slab_2d_f64", 9, 64, 64, 1, "f64", 20, geometry="slab"),
        # the 2D drop of the flux sweep, a longer stretch of steps between reads
        _run("drop_2d_f32", 9, 256, 256, 1, "f32", 50),
        # the headline: spherical drop at density ratio 10, FP32 pairs
        _run("sphere_f32", 19, 192, 192, 192, "f32", 20, gamma=10.0),
        # the same drop on the FP64 path, the one every result is compared with
        _run("sphere_f64", 19, 128, 128, 128, "f64", 4, gamma=10.0),
        # FP32 pairs with exact colour masses: the storage for small fluxes and long runs
        _run("sphere_f32x", 19, 192, 192, 192, "f32x", 10, gamma=10.0),
        # the mixed form: 16-bit recolour-on-pull populations, half the memory of a lattice
        _run("sphere_f16rc", 19, 192, 192, 192, "f16rc", 10, gamma=10.0),
        # the mixed form's second layout: 16-bit deviations per colour
        _run("sphere_f16dev", 19, 160, 160, 160, "f16dev", 10, gamma=10.0),
        # a hemisphere on a heated substrate: walls, the paper's gradient site rule, and a flux
        # field recomputed from the state every ten steps
        _run("hemisphere_heated_f32", 19, 160, 160, 160, "f32", 20, geometry="cap", walls=True,
             rule="gradient", flux="heated"),
        # a cap in a solid cup, odd sizes: ragged tiles, walls and interior solids
        _run("cavity_ragged_f32", 19, 131, 117, 89, "f32", 12, geometry="cavity", walls=True,
             rule="gradient"),
        # 64 uneven drops advanced together (48 D2Q9, 16 D3Q19), tiling from the autotuner
        {"name": "ensemble_64", "kind": "ensemble", "n2": 48, "n3": 16, "set": inputs.SEED,
         "storage": "f32", "steps": 10},
        # one iteration of the flux fit on the sessile cap at full size, FP32
        {"name": "fit_cap_f32", "kind": "fit", "nx": 256, "ny": 256, "nz": 128, "storage": "f32",
         "steps": 32, "ckpt": 32},
        # the reduced cap in FP64, on which gradients are checked by finite differences
        {"name": "fit_reduced_f64", "kind": "fit", "nx": 64, "ny": 64, "nz": 32, "storage": "f64",
         "steps": 24, "ckpt": 8},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["2d", "3d", "3d", "3d", "wall", "ensemble", "fit"])
    if kind == "2d":
        return _strip(_run("", 9, _log_int(rng, 40, 700), _log_int(rng, 40, 700), 1,
                           rng.choice(["f64", "f32", "f32", "f32x", "f16rc", "f16dev"]),
                           rng.randint(4, 50), rng.choice(["slab", "drop"]),
                           rule=rng.choice(["band", "band", "gradient"]),
                           gamma=rng.choice([1.0, 1.0, 4.0])))
    if kind == "3d":
        storage = rng.choice(["f32", "f32", "f64", "f32x", "f16rc", "f16dev"])
        hi = 120 if storage == "f64" else 192
        return _strip(_run("", 19, *(_log_int(rng, 20, hi) for _ in range(3)), storage,
                           rng.randint(2, 8 if storage == "f64" else 16),
                           rule=rng.choice(["band", "band", "gradient"]),
                           gamma=rng.choice([1.0, 2.0, 10.0])))
    if kind == "wall":
        return _strip(_run("", 19, *(_log_int(rng, 32, 176) for _ in range(3)),
                           rng.choice(["f32", "f32", "f32x", "f16dev"]), rng.randint(4, 20),
                           rng.choice(["cap", "cavity"]), walls=True, rule="gradient",
                           flux=rng.choice(["scalar", "heated"])))
    if kind == "ensemble":
        return {"kind": "ensemble", "n2": rng.randint(2, 40), "n3": rng.randint(1, 14),
                "set": rng.randint(1, 1 << 30), "storage": rng.choice(["f32", "f32", "f32x"]), "steps": rng.randint(2, 10)}
    storage = rng.choice(["f32", "f32", "f64"])
    hi = 90 if storage == "f64" else 220
    steps = rng.randint(4, 24)
    return {"kind": "fit", "nx": _log_int(rng, 40, hi), "ny": _log_int(rng, 40, hi),
            "nz": _log_int(rng, 24, hi // 2), "storage": storage, "steps": steps,
            "ckpt": rng.randint(3, steps)}


def _strip(case):
    return {k: v for k, v in case.items() if k != "name"}


# ------------------------------------------------------------------ inputs ------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _distance(shape, center):
    """Distance from center = (z, y, x) of every cell, FP64 on the GPU; a single plane is 2D."""
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") - c for n, c in zip(shape, center)]
    if shape[0] == 1:
        ax[0] = torch.zeros(1, dtype=torch.float64, device="cuda")
    return torch.sqrt(ax[0].view(-1, 1, 1) ** 2 + ax[1].view(1, -1, 1) ** 2 + ax[2].view(1, 1, -1) ** 2)


def _smallest(shape):
    return min(n for n in shape if n > 1)


def _phase(case, shape, rnd):
    """Initial phase field of a run case: a tanh interface of width 2, its place and size from the
    seed (rnd: five numbers in [0, 1))."""
    nz, ny, nx = shape
    jit = [(r - 0.5) * 3.0 for r in rnd[:3]]
    grow = 0.95 + 0.1 * rnd[3]
    mid = [(n - 1) / 2.0 + j for n, j in zip(shape, jit)]
    if case["geometry"] == "slab":
        y = torch.arange(ny, dtype=torch.float64, device="cuda").view(1, -1, 1)
        return torch.tanh((0.25 * ny * grow - (y - mid[1]).abs()) / 2.0).expand(shape).contiguous()
    if case["geometry"] == "drop":
        R0 = 32.0 / 192.0 if case["gamma"] == 10.0 else 40.0 / 256.0  # of the box side
        return torch.tanh((max(6.0, R0 * 1.6 * _smallest(shape)) * grow - _distance(shape, mid)) / 2.0)
    if case["geometry"] == "cap":
        R0 = 0.34 * min(nx, ny, 2 * nz) * grow
        return torch.tanh((R0 - _distance(shape, (-0.5, mid[1], mid[2]))) / 2.0)
    r_in, r_out, depth = _cup(shape)
    z0 = depth - 0.5 + 0.3 * r_out
    z = torch.arange(nz, dtype=torch.float64, device="cuda").view(-1, 1, 1)
    cap = torch.tanh((1.1 * r_out * grow - _distance(shape, (z0, (ny - 1) / 2.0, (nx - 1) / 2.0))) / 2.0)
    cup = torch.tanh((r_in - _axis_distance(shape)) / 2.0)
    return torch.where(z < depth, cup, cap).contiguous()


def _axis_distance(shape):
    return _distance((1,) + tuple(shape[1:]), (0.0, (shape[1] - 1) / 2.0, (shape[2] - 1) / 2.0))


def _cup(shape):
    """Inner and outer radius and depth of the solid cup on the wall z = -1/2."""
    r_in = 0.26 * min(shape[1], shape[2])
    return r_in, r_in + 3.0, max(3, min(8, shape[0] // 8))


def _solid(case, shape):
    if case["geometry"] != "cavity":
        return None
    r_in, r_out, depth = _cup(shape)
    r = _axis_distance(shape)
    ring = ((r >= r_in) & (r < r_out)).to(torch.uint8)
    out = torch.zeros(shape, dtype=torch.uint8, device="cuda")
    out[:depth] = ring
    return out


def _noise(q, shape, g):
    n = torch.rand((2, q) + tuple(shape), dtype=torch.float32, device="cuda", generator=g)
    return n.mul_(2e-6).sub_(1e-6)


def _setup(case, seed):
    """Parameters (inputs.Case), phase field, noise and solids of a run case."""
    shape = (case["nz"], case["ny"], case["nx"])
    g = _generator(seed)
    rnd = torch.rand(5, dtype=torch.float64, device="cuda", generator=g).tolist()
    paper = case["walls"]  # the paper's own drops on a wall: beta 0.99, sigma 0.1, Gamma 0.305
    band = case["rule"] == "band"
    c = inputs.Case("case", case["q"], shape, periodic=(1, 1, 0 if case["walls"] else 1),
                    rho_r_in=case["gamma"], tau_b=0.8 if case["gamma"] != 1.0 else 1.0,
                    sigma=0.1 if paper else inputs.sigma_from_amplitude(0.005 if case["q"] == 19 else 0.01),
                    beta=0.99 if paper else 0.7,
                    site_rule=inputs.RULE_BAND if band else inputs.RULE_GRADIENT,
                    threshold=0.5 if band else (0.305 if paper else 0.2),
                    phi=1e-3 if paper else 10.0 ** (-6.0 + 2.0 * rnd[4]))
    solid = _solid(case, shape)
    noise = _noise(case["q"], shape, g)
    if solid is not None:
        noise.mul_((solid == 0).to(torch.float32))
    return c, _phase(case, shape, rnd), noise, solid


def _heat_length(case):
    return 0.34 * min(case["nx"], case["ny"], 2 * case["nz"])


def _fit_setup(case, seed):
    """The flux fit on a sessile cap: the workload's geometry at this size, coefficients and the
    residual of the volume history (the weights of the gradient product) from the seed."""
    shape = (case["nz"], case["ny"], case["nx"])
    g = _generator(seed)
    R0 = 48.0 / 128.0 * min(case["nx"] / 2.0, case["ny"] / 2.0, float(case["nz"]))
    jit = ((torch.rand(3, dtype=torch.float64, device="cuda", generator=g) - 0.5) * 2.0).tolist()
    R0 *= 1.0 + 0.05 * jit[2]
    cy, cx = (shape[1] - 1) / 2.0 + jit[0], (shape[2] - 1) / 2.0 + jit[1]
    c = inputs.sessile_cap_3d(shape, R0=R0, phi0=2e-5)
    rhoN0 = torch.tanh((R0 - _distance(shape, (-0.5, cy, cx))) / 2.0)
    a = torch.randn(FIT_COEFFICIENTS, dtype=torch.float64, device="cuda", generator=g) * 0.1
    r = _distance((1,) + shape[1:], (0.0, cy, cx)) / R0
    # sites lie near the cap; the polynomial is held at its value at 1.5 R0 beyond that
    r = r.clamp(max=1.5)
    flux = torch.ones_like(r)
    for k in range(1, FIT_COEFFICIENTS + 1):
        flux = flux + a[k - 1] * r ** k
    flux = (2e-5 * flux).expand(shape).contiguous()
    resid = torch.rand(case["steps"] + 1, dtype=torch.float64, device="cuda", generator=g) + 0.5
    return c, rhoN0, flux, resid


def _members(case):
    every = inputs.ensemble_members(case["set"])
    return every[:case["n2"]] + every[48:48 + case["n3"]]


# ------------------------------------------------------------------ a pass ------------------

def _state(c, storage, rhoN0, noise, solid=None):
    sim = Sim.from_case(c, storage)
    if solid is not None:
        sim.set_solid(solid)
    sim.set_flux(c.phi)
    sim.init_equilibrium(rhoN0, noise)
    return sim


def prepare(case, seed):
    if case["kind"] == "run":
        c, rhoN0, noise, solid = _setup(case, seed)
        sim = _state(c, case["storage"], rhoN0, noise, solid)
        if case["flux"] == "heated":
            sim.set_flux_heated(c.phi, 0.5, _heat_length(case), HEATED_EVERY)
        return {"kind": "run", "sim": sim, "steps": case["steps"], "storage": case["storage"]}
    if case["kind"] == "fit":
        c, rhoN0, flux, resid = _fit_setup(case, seed)
        sim = Sim.from_case(c, case["storage"])
        flux = flux.to(torch.float64 if case["storage"] == "f64" else torch.float32)
        return {"kind": "fit", "sim": sim, "rhoN0": rhoN0, "flux": flux, "resid": resid,
                "steps": case["steps"], "ckpt": case["ckpt"]}
    cases = _members(case)
    ens = Ensemble(cases, case["storage"])
    for j, (sim, c) in enumerate(zip(ens.members, cases)):
        g = _generator(int(seed) + 7919 * (j + 1))
        sim.set_flux(c.phi)
        sim.init_equilibrium(_member_phase(c, g), _noise(c.q, c.shape, g))
    ens.autotune(probe_steps=4)
    return {"kind": "ensemble", "ens": ens, "steps": case["steps"]}


def _member_phase(c, g):
    """A member's drop, off centre by up to a cell."""
    jit = (torch.rand(3, dtype=torch.float64, device="cuda", generator=g) * 2.0 - 1.0).tolist()
    return torch.tanh((c.R0 - _distance(c.shape, tuple((n - 1) / 2.0 + d for n, d in zip(c.shape, jit)))) / 2.0)


def run(state):
    if state["kind"] == "run":
        sim = state["sim"]
        sim.step(state["steps"])
        if state["storage"] == "f64":
            m = sim.macros()
            return {"f": sim.populations(torch.float64), "rho_r": m["rho_r"], "rho_b": m["rho_b"],
                    "u": m["u"], "rhoN": m["rhoN"]}
        return {"f": sim.populations(torch.float32)}
    if state["kind"] == "fit":
        # a fit iteration: the cap as it was, the run with this flux, and the product of the
        # history's Jacobian with the residual; history and gradient in the flux's own type
        sim = state["sim"]
        sim.init_equilibrium(state["rhoN0"])
        flux = state["flux"].detach().requires_grad_(True)
        V = volume_history(sim, flux, state["steps"], state["ckpt"])
        V.backward(state["resid"])
        return {"V": V.detach().to(flux.dtype), "grad": flux.grad, "f": sim.populations(flux.dtype)}
    state["ens"].step(state["steps"])
    return [m.populations(torch.float32) for m in state["ens"].members]


# ------------------------------------------------------------------ work --------------------

def _pop_bytes(storage, q):
    """Bytes of one cell's state."""
    return {"f64": 16.0 * q, "f32": 8.0 * q, "f32x": 8.0 * q, "f16rc": 28.0 + 2.0 * (q - 1),
            "f16dev": 8.0 + 4.0 * (q - 1)}[storage]


def work(case):
    """A step reads and writes the state once and writes a site byte (and reads one under the
    gradient rule); a read-back reads the state and writes what it returns; a reverse step reads a
    recomputed state, the adjoint state and its two fields, and writes those."""
    ops = {9: 230.0, 19: 500.0}  # of one cell's update
    if case["kind"] == "run":
        n = float(case["nx"] * case["ny"] * case["nz"])
        q, s = case["q"], _pop_bytes(case["storage"], case["q"])
        step = 2 * s + (1 if case["rule"] == "band" else 2)
        step += 4 if case["flux"] == "heated" else 0
        back = s + 2 * q * (8 if case["storage"] == "f64" else 4)
        if case["storage"] == "f64":
            back += s + 48
        if case["flux"] == "heated":
            back += (case["steps"] // HEATED_EVERY) * (s + 4)
        return {"bytes": n * (case["steps"] * step + back), "flops": n * ops[q] * case["steps"]}
    if case["kind"] == "fit":
        n = float(case["nx"] * case["ny"] * case["nz"])
        real = 8 if case["storage"] == "f64" else 4
        s = _pop_bytes(case["storage"], 19)
        T, seg = case["steps"], -(-case["steps"] // case["ckpt"])
        forward = T * (2 * s + 1 + real) + seg * 2 * s
        reverse = T * (2 * s + 1 + real) + T * (3 * s + 4 * real + 17)
        ends = 8 + s + s + 38 * real
        return {"bytes": n * (forward + reverse + ends), "flops": n * T * ops[19] * 4}
    total, flops = 0.0, 0.0
    for c in _members(case):
        s = _pop_bytes(case["storage"], c.q)
        total += c.ncell * (case["steps"] * (2 * s + 1) + s + 8 * c.q)
        flops += c.ncell * case["steps"] * ops[c.q]
    return {"bytes": total, "flops": flops}


# ------------------------------------------------------------------ in 64 bits --------------

class _Plain:
    """The timestep in plain FP64 torch on whole lattices: Eq. (Stream) with halfway bounce-back,
    the sites and Eq. (exchange), moments, Eq. (cg), Eq. (collision), Eq. (perturb), Eq. (recolor)
    of the paper's Sec. II."""

    C9 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0),
          (1, -1, 0), (-1, 1, 0)]
    C19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
           (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
           (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]

    def __init__(self, c, solid=None):
        self.p, self.Q = c, c.q
        self.c = self.C9 if c.q == 9 else self.C19
        cls = [sum(v * v for v in d) for d in self.c]
        if c.q == 9:
            w, a, b, k = (4 / 9, 1 / 9, 1 / 36), (0.0, 1 / 5, 1 / 20), (1.0, -1 / 5, -1 / 20), (-4 / 27, 2 / 27, 5 / 108)
        else:
            w, a, b, k = (1 / 3, 1 / 18, 1 / 36), (0.0, 1 / 12, 1 / 24), (1.0, -1 / 12, -1 / 24), (-1 / 3, 1 / 18, 1 / 36)
        self.W, self.A, self.B, self.K = ([t[s] for s in cls] for t in (w, a, b, k))
        self.norm = [math.sqrt(s) for s in cls]
        self.opp = [0] + [i + 1 if i & 1 else i - 1 for i in range(1, self.Q)]
        w0 = w[0]
        rmin = min(c.rho_r_in, c.rho_b_in)
        self.al = [w0 if r <= rmin else 1.0 - (1.0 - w0) * rmin / r for r in (c.rho_r_in, c.rho_b_in)]
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.fluid = torch.ones(c.shape, dtype=torch.bool, device=dev) if solid is None else solid == 0
        # bounce[i]: the pull source x - c_i is solid or beyond a wall (None: nowhere)
        self.bounce = []
        for d in self.c:
            bad = self._at(~self.fluid, d) if solid is not None else torch.zeros_like(self.fluid)
            for axis, dim in ((0, 2), (1, 1), (2, 0)):
                if d[axis] and not c.periodic[axis]:
                    edge = [slice(None)] * 3
                    edge[dim] = 0 if d[axis] > 0 else -1
                    bad[tuple(edge)] = True
            self.bounce.append(bad if bool(bad.any()) else None)

    @staticmethod
    def _at(t, d):
        """The value at x - d, wrapped."""
        if d == (0, 0, 0):
            return t
        return torch.roll(t, shifts=(d[2], d[1], d[0]), dims=(-3, -2, -1))

    def start(self, rhoN0, noise):
        p, f = self.p, []
        for k, rho in enumerate((p.rho_r_in * (1 + rhoN0) / 2, p.rho_b_in * (1 - rhoN0) / 2)):
            for i in range(self.Q):
                v = rho * (self.A[i] + self.B[i] * self.al[k])
                if noise is not None:
                    v = v + noise[k, i].double()
                f.append(torch.where(self.fluid, v, torch.zeros_like(v)))
        return torch.stack(f).view((2, self.Q) + rhoN0.shape)

    def densities(self, f):
        rr, rb = f[0].sum(0), f[1].sum(0)
        return rr, rb, torch.where(self.fluid, rr + rb, torch.ones_like(rr))

    def gradient(self, rn):
        F = [torch.zeros_like(rn) for _ in range(3)]
        for i in range(1, self.Q):
            d = self.c[i]
            v = self._at(rn, tuple(-x for x in d))
            bad = self.bounce[self.opp[i]]  # x + c_i is the pull source of the opposite direction
            if bad is not None:
                v = torch.where(bad, rn, v)
            for j in range(3):
                if d[j]:
                    F[j] = F[j] + 3.0 * self.W[i] * d[j] * v
        return F

    def norm_of(self, f):
        rr, rb, rho = self.densities(f)
        F = self.gradient(torch.where(self.fluid, (rr - rb) / rho, torch.zeros_like(rr)))
        return torch.sqrt(F[0] ** 2 + F[1] ** 2 + F[2] ** 2)

    def volume(self, f):
        rr, rb, rho = self.densities(f)
        return torch.where(self.fluid, rr / rho, torch.zeros_like(rr)).sum()

    def heated(self, f, phi, K, length):
        rr, _, rho = self.densities(f)
        h = torch.where(self.fluid, rr / rho, torch.zeros_like(rr)).sum(0, keepdim=True)
        return (phi / (K + h / length)).expand(rr.shape)

    def step(self, f, phi, site=None, bulk=False):
        """One step; site: the gradient rule's sites (None: the band rule decides); bulk: hold the
        recoloring direction fixed for differentiation where one colour is a trace.  Returns the
        new state and |F|."""
        p, Q, c = self.p, self.Q, self.c
        g = []
        for k in range(2):
            for i in range(Q):
                v = self._at(f[k, i], c[i])
                if self.bounce[i] is not None:
                    v = torch.where(self.bounce[i], f[k, self.opp[i]], v)
                g.append(v)
        rr, rb = sum(g[:Q]), sum(g[Q:])
        one = torch.ones_like(rr)
        rho = torch.where(self.fluid, rr + rb, one)
        if site is None:
            site = ((rr - rb) / rho).detach().abs() < p.threshold
        e = torch.where(site & self.fluid, phi / p.sbar * one, torch.zeros_like(rr))
        fc = [g[i] + g[Q + i] for i in range(Q)]
        del g
        rr, rb = rr - e, rb + e
        wr, wb = rr / rho, rb / rho
        u = [sum(fc[i] * c[i][j] for i in range(Q) if c[i][j]) / rho if any(d[j] for d in c) else torch.zeros_like(rr)
             for j in range(3)]
        itau = wr / p.tau_r + wb / p.tau_b
        abar = wr * self.al[0] + wb * self.al[1]
        F = self.gradient(torch.where(self.fluid, (rr - rb) / rho, torch.zeros_like(rr)))
        F2 = F[0] ** 2 + F[1] ** 2 + F[2] ** 2
        pos = F2 > 0
        Fn = torch.where(pos, torch.sqrt(torch.where(pos, F2, one)), torch.zeros_like(rr))
        iF = torch.where(pos, 1.0 / torch.where(pos, Fn, one), torch.zeros_like(rr))
        trace = (wr * wb < 1e-6) if bulk else None
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        red, blue = [], []
        zero = torch.zeros_like(rr)
        for i in range(Q):
            cu = sum(c[i][j] * u[j] for j in range(3) if c[i][j]) if i else zero
            cF = sum(c[i][j] * F[j] for j in range(3) if c[i][j]) if i else zero
            rest = rho * (self.A[i] + self.B[i] * abar)
            feq = rest + rho * self.W[i] * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
            fi = fc[i] - itau * (fc[i] - feq) + 2.25 * p.sigma * itau * (self.W[i] * cF * cF * iF - self.K[i] * Fn)
            fr = wr * fi
            if i:
                cos = cF * iF / self.norm[i]
                if trace is not None:
                    cos = torch.where(trace, cos.detach(), cos)
                fr = fr + p.beta * wr * wb * cos * rest
            red.append(torch.where(self.fluid, fr, zero))
            blue.append(torch.where(self.fluid, fi - fr, zero))
        return torch.stack(red + blue).view((2, Q) + rr.shape), Fn

    def macros(self, f):
        rr, rb, rho = self.densities(f)
        tot = f[0] + f[1]
        u = torch.stack([sum(tot[i] * self.c[i][j] for i in range(self.Q) if self.c[i][j]) / rho
                         if any(d[j] for d in self.c) else torch.zeros_like(rr) for j in range(3)])
        return {"rho_r": rr, "rho_b": rb, "u": u, "rhoN": (rr - rb) / rho}


def _advance(plain, f, phi, steps, gradient, heat=None):
    Fn = plain.norm_of(f) if gradient else None
    flux = phi
    for t in range(steps):
        if heat is not None and t % HEATED_EVERY == 0:
            flux = plain.heated(f, phi, 0.5, heat)
        f, Fn = plain.step(f, flux, Fn > plain.p.threshold if gradient else None)
    return f


def exact(case, seed):
    if case["kind"] == "run":
        c, rhoN0, noise, solid = _setup(case, seed)
        plain = _Plain(c, solid)
        f = plain.start(rhoN0, noise)
        del noise
        with torch.no_grad():
            f = _advance(plain, f, c.phi, case["steps"], case["rule"] == "gradient",
                         _heat_length(case) if case["flux"] == "heated" else None)
            if case["storage"] == "f64":
                return {"f": f, **plain.macros(f)}
            return {"f": f}
    if case["kind"] == "fit":
        from torch.utils.checkpoint import checkpoint

        c, rhoN0, flux, resid = _fit_setup(case, seed)
        plain = _Plain(c)
        flux = flux.to(torch.float64 if case["storage"] == "f64" else torch.float32).double().requires_grad_(True)
        f = plain.start(rhoN0, None)
        V = [plain.volume(f)]
        for _ in range(case["steps"]):
            f = checkpoint(lambda s, phi: plain.step(s, phi, None, True)[0], f, flux, use_reentrant=False)
            V.append(plain.volume(f))
        V = torch.stack(V)
        V.backward(resid)
        return {"V": V.detach(), "grad": flux.grad, "f": f.detach()}
    out = []
    with torch.no_grad():
        for j, c in enumerate(_members(case)):
            plain = _Plain(c)
            g = _generator(int(seed) + 7919 * (j + 1))
            f = plain.start(_member_phase(c, g), _noise(c.q, c.shape, g))
            out.append(_advance(plain, f, c.phi, case["steps"], False))
    return out
