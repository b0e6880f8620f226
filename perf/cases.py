"""The work that is timed when the library is made faster.

A pass is what a program does with a state it holds on the GPU: set it, advance it by some time
steps, read the conserved functional, and take the state back (`Sim.set_spinor_device`, `step`,
`norm`, `get_spinor_device`; `batch_step` for several simulations together).  The simulations are
made once in `prepare` and kept, as a program that runs many packets through one problem keeps
them.  No launch plan is autotuned: the built-in rule is what every caller gets.

A case: dims and nx, ny, nz (cells), dx ratios ry, rz (lattice constants along y and z over the
one along x), mass m, precision, the field set, the number of time steps, and how many simulations
advance together (batch; the members differ in size, see `members`).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1309_3452_gb300 import dirac as D
from paper_1309_3452_gb300 import workloads as W

# half-lattice offsets (x, y, z) of the planes, and which of them are the upper sheet
OFFS = {3: ((0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1), (0, 0, 1), (1, 1, 1), (1, 0, 0), (0, 1, 0)),
        2: ((0, 0, 0), (1, 1, 0), (1, 0, 0), (0, 1, 0))}


def _case(name, dims, n, precision, field, steps, m=1.0, ry=1.0, rz=1.0, batch=1):
    return {"name": name, "dims": dims, "nx": n[0], "ny": n[1], "nz": n[2] if dims == 3 else 1, "ry": ry,
            "rz": rz, "m": m, "precision": precision, "field": field, "steps": steps, "batch": batch}


def listed():
    return [
        # the smallest run of the benchmark's set: (2+1)D 64^2 massless packet, 200 steps, FP64 (validation)
        _case("2d64_free_fp64", 2, (64, 64), "fp64", "free", 200, m=0.0),
        # a small ragged (2+1)D grid in a uniform vector potential, FP32: launches and latency count
        _case("2d300x260_consta", 2, (300, 260), "fp32", "const_a", 200, m=0.3),
        # (2+1)D Klein-step scattering at the benchmark's size (its 5000 steps, cut)
        _case("2d4096_klein", 2, (4096, 4096), "fp32", "klein", 120, m=0.2),
        # (2+1)D packet in a moving plane wave: fields that change with time, one step per pass
        _case("2d1000_wave", 2, (1000, 1000), "fp32", "wave", 100),
        # the benchmark's (3+1)D 128^3 free packet (its 1000 steps, cut)
        _case("3d128_free", 3, (128, 128, 128), "fp32", "free", 100),
        # an odd-sized anisotropic (3+1)D grid with a Klein step, of the serving stream's sizes
        _case("3d203_klein_aniso", 3, (203, 149, 91), "fp32", "klein", 60, m=0.45, ry=1.2, rz=0.9),
        # the benchmark's headline: (3+1)D 512^3, soft core and moving plane wave (its 2000 steps, cut)
        _case("3d512_laser", 3, (512, 512, 512), "fp32", "laser", 16),
        # absorbing layers around a uniform region: a coefficient for every value
        _case("3d160_layers", 3, (160, 160, 160), "fp32", "layers", 50),
        # an arbitrary static vector potential given by its link integrals
        _case("3d128_links", 3, (128, 128, 128), "fp32", "links", 40),
        # the FP64 validation runs beside the FP32 ones: free, and the laser's fields
        _case("3d96_free_fp64", 3, (96, 96, 96), "fp64", "free", 40),
        _case("3d64_laser_fp64", 3, (64, 64, 64), "fp64", "laser", 20),
        # one quantum of the serving loop: residents of many sizes, both dimensions, stepped together
        _case("serve_8", 3, (160, 160, 160), "fp32", "mixed", 100, m=0.5, batch=8),
    ]


def draw(rng):
    """A case of the same ranges: the field sets and precisions above over the serving stream's and the
    benchmark's sizes (sides log-uniform, odd ones among them), 10 to 200 steps, no more site updates
    than about half a second of work at the start."""
    dims = rng.choice((2, 3, 3))
    precision = rng.choice(("fp32", "fp32", "fp32", "fp64"))
    lo, hi = ((64, 4096) if dims == 2 else (32, 384)) if precision == "fp32" else ((48, 1024) if dims == 2 else (16, 128))
    n = [int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) for _ in range(3)]
    if rng.random() < 0.4:  # cubes and squares are as common as anything
        n = [n[0]] * 3
    if precision == "fp32" and rng.random() < 0.15:
        return _case("", 3, [min(n[0], 200)] * 3, precision, "mixed", rng.randint(20, 100), round(rng.random(), 3),
                     batch=rng.randint(2, 10))
    fields = ["free", "klein", "const_a", "wave", "laser", "softcore", "layers"]
    if n[0] * n[1] * (n[2] if dims == 3 else 1) < 4e6:
        fields.append("links")
    field = rng.choice(fields)
    cells = n[0] * n[1] * (n[2] if dims == 3 else 1)
    budget = (2e9 if dims == 3 else 5e9) if precision == "fp32" else 1.5e7
    steps = max(4, min(rng.randint(10, 200), int(budget / cells)))
    iso = field == "laser" or rng.random() < 0.6
    return _case("", dims, n, precision, field, steps, round(rng.random(), 3), 1.0 if iso else round(rng.uniform(0.9, 1.3), 2),
                 1.0 if iso else round(rng.uniform(0.9, 1.3), 2), 1)


def members(case):
    """The problems of a case: one, or (batch) residents of sizes down to a fifth of the case's, (3+1)D
    and (2+1)D (four times the side) in turn, half of them with a Klein step, as the serving stream has them."""
    if case["batch"] == 1:
        return [case]
    out = []
    for i in range(case["batch"]):
        side = max(16, int(case["nx"] * (1.0 - 0.8 * i / case["batch"])))
        dims = 3 if i % 2 == 0 else 2
        s = side if dims == 3 else 4 * side
        out.append(dict(case, batch=1, dims=dims, nx=s, ny=s, nz=s if dims == 3 else 1, ry=1.0, rz=1.0,
                        field="klein" if i % 4 < 2 else "free"))
    return out


def fields_of(c):
    """The field parameters of one problem, as plain values (lengths in units of the lattice constant along x)."""
    n = (c["nx"], c["ny"], c["nz"])
    dx = (1.0, c["ry"], c["rz"])
    ctr = tuple(n[a] * dx[a] / 2.0 for a in range(3))
    f = c["field"]
    out = {}
    if f == "klein":
        out = dict(step_axis=0, step_x0=n[0] / 2.0 + 0.25, step_V=0.5 + c["m"])
    elif f == "const_a":
        out = dict(q=0.8, A_const=(0.3, -0.45, 0.2 if c["dims"] == 3 else 0.0))
    if f in ("wave", "laser"):  # travels along the last axis, polarised along x
        a = c["dims"] - 1
        k = [0.0, 0.0, 0.0]
        k[a] = 2.0 * math.pi / (n[a] * dx[a]) * max(1, n[a] // 64)
        out = dict(q=1.0, Apw_amp=0.5, Apw_k=tuple(k), Apw_omega=k[a], Apw_pol=0)
    if f in ("softcore", "laser"):
        out |= dict(sc_Z=1.0, sc_a=1.0, sc_center=(ctr[0], ctr[1], ctr[2] if c["dims"] == 3 else 0.0))
    if f == "layers":
        out = dict(V0=0.05, abs_W=0.7, abs_width=max(3.0, n[0] / 10.0), abs_axes=(1 << c["dims"]) - 1)
    return out


def _links(c, seed):
    shape = (c["dims"], len(OFFS[c["dims"]]), c["nz"], c["ny"], c["nx"])
    return 0.3 * (2.0 * np.random.default_rng(seed + 77).random(shape) - 1.0)


def _dt(c):
    """0.9 of the stability bound sum (dt/dx_a)^2 <= 1."""
    s = 1.0 + 1.0 / c["ry"] ** 2 + (1.0 / c["rz"] ** 2 if c["dims"] == 3 else 0.0)
    return 0.9 / math.sqrt(s)


def _problem(c, seed):
    f = W.Fields(**fields_of(c), **({"A_links": _links(c, seed)} if c["field"] == "links" else {}))
    return W.Problem(c["dims"], (c["nx"], c["ny"], c["nz"]), (1.0, c["ry"], c["rz"] if c["dims"] == 3 else 1.0), _dt(c),
                     c["m"], f)


def _packet(c, seed):
    """A Gaussian packet with a seeded momentum, width and place (complex128, canonical layout, on the GPU),
    normalised; the planes hold the continuum spinor's components at their own points and sheet times."""
    rng = np.random.default_rng(seed)
    dims = c["dims"]
    n, dx = (c["nx"], c["ny"], c["nz"]), (1.0, c["ry"], c["rz"])
    L = [n[a] * dx[a] for a in range(dims)]
    klein = c["field"] == "klein"
    k = rng.random() * (lambda d: d / np.linalg.norm(d))(rng.standard_normal(3))
    k = [float(v) for v in k[:dims]]
    ctr = [L[a] * ((0.25 if klein and a == 0 else 0.5) + 0.05 * (rng.random() - 0.5)) for a in range(dims)]
    sigma = min(L) / 8.0 * (0.8 + 0.4 * rng.random())
    E = math.sqrt(c["m"] ** 2 + sum(v * v for v in k))
    kz = k[2] if dims == 3 else 0.0
    w = [E + c["m"], 0.0, kz, k[0] + 1j * k[1]] if dims == 3 else [E + c["m"], k[0] + 1j * k[1]]
    out = torch.empty((len(OFFS[dims]), c["nz"], c["ny"], c["nx"]), dtype=torch.complex128, device="cuda")
    for p, o in enumerate(OFFS[dims]):
        fac = []
        for a in range(3):
            if a >= dims:
                fac.append(torch.ones(1, dtype=torch.complex128, device="cuda"))
                continue
            x = (torch.arange(n[a], dtype=torch.float64, device="cuda") + 0.5 * o[a]) * dx[a]
            d = x - ctr[a]
            d = d - L[a] * torch.round(d / L[a])
            fac.append(torch.polar(torch.exp(-d * d / (2 * sigma * sigma)), k[a] * x))
        t = -0.5 * _dt(c) if p < len(OFFS[dims]) // 2 else 0.0
        s = w[p // 2] * np.exp(-1j * E * t)
        torch.mul((fac[1][:, None] * fac[0][None, :])[None], (fac[2] * complex(s))[:, None, None], out=out[p])
    total = sum(float(torch.view_as_real(out[p]).square().sum()) for p in range(len(out)))
    return out.mul_(1.0 / math.sqrt(total))


def prepare(case, seed):
    sims, psi, out = [], [], []
    for i, c in enumerate(members(case)):
        psi.append(_packet(c, seed + 1000 * i))
        out.append(torch.empty_like(psi[-1]))
        sims.append(D.Sim(_problem(c, seed + 1000 * i), D.FP32 if c["precision"] == "fp32" else D.FP64))
    return {"sims": sims, "psi": psi, "out": out, "steps": case["steps"]}


def run(state):
    sims = state["sims"]
    for s, p in zip(sims, state["psi"]):
        s.time = 0.0
        s.set_spinor_device(p.data_ptr())
    if len(sims) == 1:
        sims[0].step(state["steps"])
    else:
        D.batch_step(sims, state["steps"])
    E = [s.norm() for s in sims]
    for s, o in zip(sims, state["out"]):
        s.get_spinor_device(o.data_ptr())
    return {"psi": state["out"], "E": [e[0] for e in E], "naive": [e[1] for e in E]}


def work(case):
    """Bytes: the complex128 state in and out once, and the given per-value data once.  Flops: per value
    and half-step three complex differences (6), their sum (4) and the Cayley update (14), a link factor
    two complex products more per axis (12)."""
    b = f = 0.0
    for c in members(case):
        values = float(c["nx"] * c["ny"] * c["nz"] * len(OFFS[c["dims"]]))
        b += values * (32.0 + (8.0 * c["dims"] if c["field"] == "links" else 0.0))
        axes = {"const_a": c["dims"], "links": c["dims"], "wave": 1, "laser": 1}.get(c["field"], 0)
        f += values * case["steps"] * (14.0 + 2.0 * c["dims"] + 2.0 * (c["dims"] - 1) + 12.0 * axes)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64-bit values in plain torch
class _Plain:
    """The scheme (arXiv:1309.3452, Eqs. ss1-ss4) on whole complex128 planes."""

    def __init__(self, c, seed):
        self.c, self.dims, self.off = c, c["dims"], OFFS[c["dims"]]
        self.P = len(self.off)
        self.n = (c["nx"], c["ny"], c["nz"])
        self.dx = (1.0, c["ry"], c["rz"])
        self.dt = _dt(c)
        self.f = fields_of(c)
        self.psi = _packet(c, seed)
        self.links = torch.from_numpy(_links(c, seed)).cuda() if c["field"] == "links" else None

    def coord(self, p, a, shift=0.0):
        """Coordinates along axis a of plane p's points, shaped to broadcast over (z, y, x)."""
        x = (torch.arange(self.n[a], dtype=torch.float64, device="cuda") + 0.5 * self.off[p][a] + shift) * self.dx[a]
        return x.view([-1 if 2 - a == d else 1 for d in range(3)])

    def potential(self, p):
        """V at plane p's points (complex where there are layers), broadcastable."""
        f = self.f
        V = torch.full((1, 1, 1), f.get("V0", 0.0), dtype=torch.float64, device="cuda")
        if "step_axis" in f:
            V = V + f["step_V"] * (self.coord(p, f["step_axis"]) > f["step_x0"]).double()
        if "sc_Z" in f:
            r2 = f["sc_a"] ** 2
            for a in range(self.dims):
                r2 = r2 + (self.coord(p, a) - f["sc_center"][a]) ** 2
            V = V - f["sc_Z"] / torch.sqrt(r2)
        if "abs_W" in f:
            w = torch.zeros((1, 1, 1), dtype=torch.float64, device="cuda")
            for a in range(self.dims):
                x = self.coord(p, a)
                d = torch.minimum(x, self.n[a] * self.dx[a] - x)
                w = w + torch.where(d < f["abs_width"], (1.0 - d / f["abs_width"]) ** 2, torch.zeros_like(d))
            V = torch.complex(V.expand(w.shape).contiguous(), -f["abs_W"] * w)
        return V

    def partner(self, p, a):
        o = list(self.off[p])
        o[a] ^= 1
        return self.off.index(tuple(o))

    def phase(self, p, a, down, t):
        """q times the line integral of A over the link from plane p's points up (or, from the lower
        neighbour's point up to them) along axis a, at time t; None where there is no vector potential."""
        f, h = self.f, 0.5 * self.dx[a]
        if self.links is not None:
            if not down:
                return self.links[a, p]
            q = self.links[a, self.partner(p, a)]  # the lower neighbour's up link
            return torch.roll(q, 1, 2 - a) if self.off[p][a] == 0 else q
        if "A_const" in f:
            return torch.full((1, 1, 1), f["q"] * f["A_const"][a] * h, dtype=torch.float64, device="cuda")
        if "Apw_amp" in f and f["Apw_pol"] == a:
            k = self.dims - 1  # the wave vector's axis, across the polarisation
            ph = f["Apw_k"][k] * self.coord(p, k) - f["Apw_omega"] * t
            return f["q"] * f["Apw_amp"] * h * torch.cos(ph)
        return None

    def neighbour(self, psi, p, a, up):
        q = psi[self.partner(p, a)]
        if self.off[p][a] == 0:
            return q if up else torch.roll(q, 1, 2 - a)
        return torch.roll(q, -1, 2 - a) if up else q

    def S(self, psi, p, t):
        odd = (self.off[p][0] + self.off[p][1]) % 2
        total = None
        for a in range(self.dims):
            up, dn = self.neighbour(psi, p, a, True), self.neighbour(psi, p, a, False)
            pu = self.phase(p, a, False, t)
            if pu is not None:
                pd = self.phase(p, a, True, t)
                up = up * torch.polar(torch.ones_like(pu), -pu)
                dn = dn * torch.polar(torch.ones_like(pd), pd)
            s = (1.0, 1j if odd else -1j, -1.0 if odd else 1.0)[a] * (self.dt / self.dx[a])
            d = (up - dn).mul_(s)
            total = d if total is None else total.add_(d)
        return total

    def step(self, t):
        half = self.P // 2
        for upper in (True, False):
            new = []
            for p in range(half) if upper else range(half, self.P):
                th = 0.5 * self.dt * ((1.0 if upper else -1.0) * self.c["m"] + self.V[p])
                S = self.S(self.psi, p, t if upper else t + 0.5 * self.dt)
                new.append(((1.0 - 1j * th) * self.psi[p] - S) / (1.0 + 1j * th))
            for i, v in enumerate(new):
                self.psi[i if upper else half + i].copy_(v)
            del new

    def run(self, steps):
        self.V = [self.potential(p) for p in range(self.P)]
        for i in range(steps):
            self.step(i * self.dt)
        return self

    def functional(self, t):
        """(E, sum |psi|^2): E = sum |psi|^2 + Re sum over the lower values of conj(G) S_G, links at t - dt/2."""
        naive = sum(float(torch.view_as_real(v).square().sum()) for v in self.psi)
        cross = 0.0
        for p in range(self.P // 2, self.P):
            cross += float((self.psi[p].conj() * self.S(self.psi, p, t - 0.5 * self.dt)).real.sum())
        return naive + cross, naive


def exact(case, seed):
    psi, E, naive = [], [], []
    for i, c in enumerate(members(case)):
        r = _Plain(c, seed + 1000 * i).run(case["steps"])
        e, n = r.functional(case["steps"] * r.dt)
        psi.append(r.psi)
        E.append(e)
        naive.append(n)
        del r
    return {"psi": psi, "E": E, "naive": naive}
