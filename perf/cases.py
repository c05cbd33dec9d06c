"""Measured cases of the CSPH library: what a user of `Simulation`, the batched ensembles, the reverse mode and the
Voronoi balancing has it do, from a 400-particle shock tube to the 1.125M-particle plate impact, in both precisions,
with the per-step cell search and with Verlet lists.

A case is a dict of plain values.  Its kind says which entry points a pass calls:
  step      sph_step over a number of steps (optionally the FP64 totals after them)
  ensemble  one CUDA graph of several steps over a handle of independent instances of uneven size
  adjoint   a differentiable run, forward and reverse
  balance   one update of the Voronoi decomposition: assignment, rates (loads, adjacency), balancing displacement

Runs with the per-step search are stepped from the same start on every pass (the caller's arrays live in one block,
restored by one copy), as a parameter study does.  Runs with Verlet lists go on from where the last pass ended, as a
simulation does, since their lists outlive a call; after `cycle` passes they start again, so that every pass stays
inside the window that the workload is meant for.

`exact` is the same mathematics in plain FP64 torch: brute cell search, pair fluxes, kick-drift-kick, autograd.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import synth

DEV = "cuda:0"
A = 1e-4                     # lattice spacing of the plates (0.1 mm)
FIELDS = ("x", "y", "z", "vx", "vy", "vz", "rho", "E", "ax", "ay", "az", "drho", "dE", "d", "P", "c")


# ---------------------------------------------------------------------------------------------- cases
def _step(name, shape, **kw):
    c = dict(name=name, kind="step", shape=shape, precision="mixed", beta=0.0, units=0, n_upd=10, order=1,
             kernel="cubic", solver="acoustic", totals=False)
    c["cycle"] = 1 if not kw.get("beta") else 4 if shape == "droplets" else 20
    c.update(kw)
    return c


def listed():
    return [
        # the 400-particle Sod tube of the accuracy tests: the smallest call, four 1D work units balanced twice in 20 steps
        _step("sod_400_fp64", "sod", precision="fp64", units=4, steps=20),
        # a small plate impact as a parameter study steps it: lists, work units, 31.7k particles
        _step("plate_32k_lists", "plate", proj=16, tx=48, tz=12, beta=0.15, units=8, steps=5),
        # the benchmark: 1.125M-particle plate impact, 64 work units, lists with buffer 0.15; output every 5 steps
        _step("plate_1125k_lists", "plate", proj=50, tx=200, tz=25, beta=0.15, units=64, steps=5),
        # the library's defaults (no lists, no work units, mixed precision) on the 387k plate
        _step("plate_387k_search", "plate", proj=30, tx=120, tz=25, steps=3),
        # the plain FP64 step every mixed result is held against, 203k plate
        _step("plate_203k_fp64", "plate", proj=25, tx=120, tz=13, precision="fp64", steps=1),
        # two Tait droplets in gas at 1:1000 density, 256 work units in 3D, totals printed with every output
        _step("droplets_1m_lists", "droplets", n_sphere=400_000, n_gas=200_000, beta=0.15, units=256, steps=5,
              totals=True),
        # grooved lead sample on a rigid wall (Mie-Grueneisen) in FP64 with lists
        _step("ejecta_65k_fp64_lists", "ejecta", nx=50, nz=10, precision="fp64", beta=0.15, steps=2),
        # second-order states, Wendland kernel and HLL solver on a plate in a plane, ragged size
        _step("plate_2d_order2", "plate_2d", proj=151, tx=603, tz=83, order=2, kernel="wendland_c2", solver="hll", steps=3),
        # batched ensemble of uneven plate impacts in one CUDA graph
        dict(name="ensemble_24_graph", kind="ensemble", count=24, n_min=5_000, n_max=200_000, beta=0.15, steps=5,
             cycle=20),
        # gradients of a short impact: FP32 forward, FP64 pair derivatives (the default of the reverse mode)
        dict(name="adjoint_32k_fp64", kind="adjoint", proj=16, tx=48, tz=12, steps=6, every=3, reverse="fp64"),
        # the same with FP32 pair derivatives on the 203k plate of the differentiable-impact configuration
        dict(name="adjoint_203k_fp32", kind="adjoint", proj=25, tx=120, tz=13, steps=4, every=2, reverse="fp32"),
        # the three-unit disk of the balancing test: one update of the decomposition
        dict(name="balance_disk_131k", kind="balance", n=127_230, K=3),
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def _plate_of(rng, lo, hi):
    """A plate impact of about N particles, N log-uniform in [lo, hi], with a ragged aspect ratio."""
    n = _log(rng, lo, hi)
    p = max(4, int(round((n / 9.0) ** (1 / 3) * rng.uniform(0.85, 1.15))))
    tz = max(3, int(round(p * rng.uniform(0.4, 0.7))))
    tx = max(p + 2, int(round(math.sqrt(max(n - p ** 3, n / 3) / tz))))
    return dict(proj=p, tx=tx, tz=tz)


def draw(rng):
    kind = rng.choice(["sod", "lists", "lists", "search", "fp64", "fp64", "droplets", "ejecta", "plane", "ensemble",
                       "adjoint", "balance"])
    if kind == "sod":
        return _unnamed(_step("", "sod", precision=rng.choice(["fp64", "mixed"]), order=rng.choice([1, 1, 2]),
                              steps=rng.randrange(10, 50), cfl=round(rng.uniform(0.15, 0.3), 4)))
    if kind == "lists":
        return _unnamed(_step("", "plate", **_plate_of(rng, 3e3, 1e6), beta=round(rng.uniform(0.1, 0.16), 3),
                              units=rng.choice([0, 0, 8, 32, 64]), steps=rng.randrange(3, 6)))
    if kind == "search":
        return _unnamed(_step("", "plate", **_plate_of(rng, 2e3, 6e5), kernel=rng.choice(["cubic", "wendland_c2"]),
                              solver=rng.choice(["acoustic", "acoustic", "hll"]), steps=rng.randrange(1, 4)))
    if kind == "fp64":
        return _unnamed(_step("", "plate", precision="fp64", **_plate_of(rng, 2e3, 2e5), beta=rng.choice([0.0, 0.0, 0.15]),
                              kernel=rng.choice(["cubic", "wendland_c2"]), order=1,
                              solver=rng.choice(["acoustic", "acoustic", "hll"]), steps=1))
    if kind == "droplets":
        n = int(_log(rng, 5e3, 4e5))
        return _unnamed(_step("", "droplets", n_sphere=n, n_gas=n // 2, beta=rng.choice([0.0, 0.15]),
                              units=rng.choice([0, 16, 64]), steps=rng.randrange(2, 5), totals=True))
    if kind == "ejecta":
        return _unnamed(_step("", "ejecta", nx=rng.randrange(24, 80), nz=rng.randrange(4, 24), beta=0.15,
                              precision=rng.choice(["mixed", "mixed", "fp64"]), steps=rng.randrange(1, 4)))
    if kind == "plane":
        p = int(_log(rng, 15, 180))
        return _unnamed(_step("", "plate_2d", proj=p, tx=4 * p + rng.randrange(9), tz=max(4, p // 2 + rng.randrange(5)),
                              precision=rng.choice(["mixed", "fp64"]), order=rng.choice([1, 2]),
                              kernel=rng.choice(["cubic", "wendland_c2"]), steps=rng.randrange(1, 5)))
    if kind == "ensemble":
        return dict(kind="ensemble", count=rng.randrange(3, 24), n_min=rng.randrange(1_000, 6_000),
                    n_max=rng.randrange(20_000, 150_000), beta=rng.choice([0.0, 0.15]), steps=rng.randrange(2, 5), cycle=20)
    if kind == "adjoint":
        steps = rng.randrange(2, 6)
        return dict(kind="adjoint", **_plate_of(rng, 3e3, 6e4), steps=steps, every=rng.randrange(1, steps + 1),
                    reverse=rng.choice(["fp64", "fp64", "fp32"]))
    return dict(kind="balance", n=int(_log(rng, 4e3, 1.3e5)), K=rng.choice([3, 5, 9, 17, 40]))


def _unnamed(c):
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------------------------------------- inputs
def _problem(c, seed):
    s = int(seed) + 1
    if c["kind"] == "balance":
        D = synth.disk(c["n"], 0.45, 0.1)
        n, a = len(D["x"]), D["a"]
        u = synth.uniform(s, 4 * n)
        pos = {k: D[k] + 0.05 * a * (2.0 * u[q::4] - 1.0) for q, k in enumerate("xyz")}
        zero = np.zeros(n)
        return synth.Problem("disk", 3, dict(pos, vx=zero, vy=zero, vz=zero, rho=np.ones(n), E=1.0 + 0.1 * u[3::4],
                                             m=np.full(n, a ** 3)),
                             [synth.MaterialSpec("ideal", 1.4)], units=c["K"], unit_dim=2)
    shape = c.get("shape", "plate")
    if shape == "sod":
        q = synth.sod_1d(seed=s)
        q.cfl = c.get("cfl", q.cfl)
    elif shape == "plate":
        q = synth.plate_impact(c["proj"], (c["tx"], c["tx"], c["tz"]), a=A, v=1000.0, seed=s, jitter=0.05)
    elif shape == "plate_2d":
        q = synth.plate_impact_2d(c["proj"], (c["tx"], c["tz"]), a=A, v=1000.0, seed=s, jitter=0.05)
    elif shape == "droplets":
        q = synth.droplets(c["n_sphere"], c["n_gas"], seed=s)
    else:
        q = synth.ejecta(nx=c["nx"], nz=c["nz"])
        u = synth.uniform(s, 3 * q.n)
        for k, ax in enumerate("xyz"):
            q.arrays[ax] = q.arrays[ax] + 0.05 * q.meta["a"] * (2.0 * u[k::3] - 1.0)
    q.units = c.get("units", 0)
    q.kernel = c.get("kernel", "cubic")
    if q.kernel == "wendland_c2":
        q.kappa = 1.936
    return q


def _ensemble(c, seed):
    """Plate impacts of log-spaced size; impact speeds, EOS gammas and the lattice jitter from the seed."""
    u = synth.uniform(int(seed) + 1, 2 * c["count"])
    out = []
    for b in range(c["count"]):
        n = c["n_min"] * (c["n_max"] / c["n_min"]) ** ((b * 7 % c["count"] + 0.5) / c["count"])
        p = max(4, int(round((n / 9.0) ** (1.0 / 3.0))))
        out.append(synth.plate_impact(p, (4 * p, 4 * p, max(p // 2, 2)), a=A, v=500.0 + 1500.0 * u[2 * b],
                                      gamma=1.5 + 1.5 * u[2 * b + 1], units=0, seed=int(seed) + 1000 * b + 7, jitter=0.05))
    return out


def _into_block(sim):
    """Lay the caller's arrays in one block of device memory (SoA views), so that one copy restores all of them."""
    keys = [k for k, v in sim.t.items() if v is not None]
    at, total = {}, 0
    for k in keys:
        at[k] = total
        total += sim.t[k].numel() * sim.t[k].element_size()
        total += -total % 8
    gen_at, total = total, total + (sim.gen.numel() * 8 if sim.gen is not None else 0)
    block = torch.zeros(total, dtype=torch.uint8, device=DEV)
    for k in keys:
        t = sim.t[k]
        view = block[at[k]: at[k] + t.numel() * t.element_size()].view(t.dtype)
        view.copy_(t)
        sim.t[k] = view
    if sim.gen is not None:
        block[gen_at:].view(torch.float64).copy_(sim.gen.reshape(-1))
    return block, gen_at


def prepare(case, seed):
    from paper_1805_05128_gb300 import Simulation, ensemble
    kind = case["kind"]
    if kind == "ensemble":
        probs = _ensemble(case, seed)
        sim = Simulation(probs, precision="mixed", units=0, cell_beta=case["beta"], cell_cap=ensemble.cell_cap(probs),
                         device=DEV)
        st = _ready(case, sim)
        st["graph"] = ensemble.GraphRun(sim, case["steps"])
        return st
    if kind == "adjoint":
        q = _problem(case, seed)
        a = {k: torch.as_tensor(v, device=DEV) for k, v in q.arrays.items()}
        f64 = dict(dtype=torch.float64, device=DEV)
        return dict(case=case, pos=torch.stack([a["x"], a["y"], a["z"]], 1), vel=torch.stack([a["vx"], a["vy"], a["vz"]], 1),
                    rho=a["rho"].clone(), E=a["E"].clone(), m=a["m"].clone(), c0=torch.tensor(5300.0, **f64),
                    gamma=torch.tensor(2.0, **f64), weight=_loss_weight(a["vz"]))
    q = _problem(case, seed)
    if kind == "balance":
        gen = _disk_generators(case["K"])
        sim = Simulation(q, precision="fp64", generators=gen, n_upd=0, device=DEV)
        return dict(case=case, sim=sim, gen0=sim.gen.clone())
    gen = synth.problem_generators(q) if case["units"] else None
    sim = Simulation(q, precision=case["precision"], units=case["units"], generators=gen, n_upd=case["n_upd"],
                     cell_beta=case["beta"], order=case["order"], solver=case["solver"], device=DEV)
    if case["units"]:
        sim.assign()
        sim.build_cells()
    return _ready(case, sim)


def _ready(case, sim):
    """Rates evaluated, and a copy of the caller's arrays to start again from."""
    block, at = _into_block(sim)
    sim.eval_rates()
    start = block.clone()
    return dict(case=case, sim=sim, block=block, start=start, passes=0,
                gen0=start[at:].view(torch.float64).view_as(sim.gen) if sim.gen is not None else None)


def _loss_weight(vz):
    """Weights of the mean axial velocity of the projector."""
    w = (vz < 0).to(torch.float64)
    return w / w.sum()


def _disk_generators(K):
    """Three off-centre generators as in the disk test, or K of them on a sunflower spiral pushed off centre."""
    if K == 3:
        return np.array([[0.0, 0.1], [-0.12, -0.25], [0.12, -0.25]])
    k = np.arange(K)
    r, t = 0.33 * np.sqrt((k + 0.5) / K), 2.399963 * k
    return np.stack([0.05 + r * np.cos(t), -0.04 + r * np.sin(t)], 1)


# ---------------------------------------------------------------------------------------------- one pass
def run(st):
    case = st["case"]
    if case["kind"] == "adjoint":
        from paper_1805_05128_gb300.adjoint import RunSpec, csph_run
        leaf = {k: st[k].detach().clone().requires_grad_() for k in ("pos", "vel", "rho", "E", "c0", "gamma")}
        spec = RunSpec(m=st["m"], n_steps=case["steps"], every=case["every"], reverse=case["reverse"])
        pos, vel, rho, E = csph_run(leaf["pos"], leaf["vel"], leaf["rho"], leaf["E"], leaf["c0"], leaf["gamma"], spec)
        (vel[:, 2] * st["weight"]).sum().backward()
        return dict(pos=pos.detach(), vel=vel.detach(), rho=rho.detach(), E=E.detach(),
                    grad={k: v.grad for k, v in leaf.items()})
    sim = st["sim"]
    if case["kind"] == "balance":
        sim.gen.copy_(st["gen0"])
        offsets = sim.assign()
        sim.eval_rates()
        shift = sim.balance()
        return dict(gen=sim.gen, shift=shift, offsets=offsets, unit=sim.t["unit"],
                    rates={k: sim.t[k] for k in ("ax", "ay", "az", "drho", "dE")})
    if st["passes"] % case["cycle"] == 0 and st["passes"]:
        st["block"].copy_(st["start"])
        if st["gen0"] is not None:
            sim.gen.copy_(st["gen0"])
    st["passes"] += 1
    if case["kind"] == "ensemble":
        st["graph"].replay()
        return _outputs(sim)
    sim.step(case["steps"])
    out = _outputs(sim)
    if case["totals"]:
        out["totals"] = sim.conservation()
    return out


def _outputs(sim):
    out = {k: sim.t[k] for k in FIELDS if sim.t[k] is not None}
    out["id"] = sim.t["id"]
    if sim.gen is not None:
        out["gen"] = sim.gen
        out["unit"] = sim.t["unit"]
    return out


# ---------------------------------------------------------------------------------------------- work of a pass
def _count(c):
    """(particles, dimension, neighbours of a lattice particle) of a case."""
    if c["kind"] == "ensemble":
        n = 0
        for b in range(c["count"]):
            nb = c["n_min"] * (c["n_max"] / c["n_min"]) ** ((b * 7 % c["count"] + 0.5) / c["count"])
            p = max(4, int(round((nb / 9.0) ** (1.0 / 3.0))))
            n += p ** 3 + 16 * p * p * max(p // 2, 2)
        return n, 3, 80
    if c["kind"] == "balance":
        return int(c["n"]), 3, 80
    shape = c.get("shape", "plate")
    if shape == "sod":
        return 400, 1, 4
    if shape == "plate_2d":
        return c["proj"] ** 2 + c["tx"] * c["tz"], 2, 20
    if shape == "droplets":
        return 2 * c["n_sphere"] + c["n_gas"], 3, 80
    if shape == "ejecta":
        return int(2 * 80 * c["nz"] * (c["nx"] - 10)), 3, 80
    return c["proj"] ** 3 + c["tx"] ** 2 * c["tz"], 3, 80


def work(case):
    """State in (14 FP64 arrays in 3D) and out (16) once per pass; 70 flops per interacting half pair and step (110 with
    reconstructed states), 60 per particle and step; the reverse mode replays the steps and costs twice a step more."""
    n, dim, nb = _count(case)
    steps = case.get("steps", 1)
    arrays_in, arrays_out = 5 + 3 * dim, 7 + 3 * dim
    pair, bytes_ = 70.0, 8.0 * n * (arrays_in + arrays_out)
    if case.get("order", 1) == 2:
        pair = 110.0
    flops = steps * n * (60.0 + pair * nb / 2)
    if case["kind"] == "adjoint":
        flops *= 4
        bytes_ = 8.0 * n * (9 + 8 + 8)
    if case["kind"] == "balance":
        flops += 6.0 * n * case["K"]
    return dict(bytes=bytes_, flops=flops)


# ---------------------------------------------------------------------------------------------- the same in plain FP64
def _t(v):
    return torch.as_tensor(np.asarray(v, dtype=np.float64), device=DEV)


class _Exact:
    """The method on one instance: x, v (n x dim), rho, E, m (n) and a material index per particle."""

    def __init__(self, q, order=1, solver="acoustic", gamma=None, c0=None):
        ax = "xyz"[: q.dim]
        self.q, self.dim, self.order, self.solver = q, q.dim, order, solver
        self.kh = 0.5 * q.kappa * q.eta
        self.x = torch.stack([_t(q.arrays[k]) for k in ax], 1)
        self.v = torch.stack([_t(q.arrays["v" + k]) for k in ax], 1)
        self.rho, self.E, self.m = (_t(q.arrays[k]) for k in ("rho", "E", "m"))
        self.mat = None if q.mat is None else torch.as_tensor(q.mat, device=DEV)
        self.par = (gamma, c0)
        self.t, self.rates = 0.0, None
        self.load = self.adj = None          # unit statistics: directed pairs per unit, adjacency
        self.unit = self.id = None
        n = len(self.rho)
        self.id = torch.arange(n, device=DEV)

    def permute(self, o):
        for k in ("x", "v", "rho", "E", "m", "mat", "unit", "id", "d", "P", "c"):
            t = getattr(self, k, None)
            if t is not None:
                setattr(self, k, t[o])
        if self.rates is not None:
            self.rates = tuple(r[o] for r in self.rates)

    def eos(self, rho, e):
        P, c2 = torch.zeros_like(rho), torch.zeros_like(rho)
        for k, mt in enumerate(self.q.materials):
            g = self.par[0] if self.par[0] is not None else mt.gamma
            if mt.eos == "ideal":
                p = (g - 1) * rho * e
                s = g * p / rho
            elif mt.eos == "stiffened":
                pinf = mt.p_inf if self.par[1] is None else mt.rho0 * self.par[1] ** 2 / g
                p = (g - 1) * rho * e - g * pinf
                s = g * (p + pinf) / rho
            elif mt.eos == "tait":
                r = rho / mt.rho0
                p = mt.rho0 * mt.c0 ** 2 / g * (r ** g - 1)
                s = mt.c0 ** 2 * r ** (g - 1)
            else:
                xx = mt.rho0 / rho
                u = 1 - xx
                D = 1 - mt.s_a * u
                ca2, du = mt.c0 ** 2, xx / rho
                Pr, er = mt.rho0 * ca2 * u / D ** 2, 0.5 * ca2 * u * u / D ** 2
                dPr, der = mt.rho0 * ca2 * (1 + mt.s_a * u) / D ** 3 * du, ca2 * u / D ** 3 * du
                p = Pr + g * rho * (e - er)
                s = dPr + g * (e - er) - g * rho * der + g * p / rho
            if len(self.q.materials) == 1:
                P, c2 = p, s
            else:
                P, c2 = torch.where(self.mat == k, p, P), torch.where(self.mat == k, s, c2)
        return P, torch.where(c2 > 0, c2, torch.zeros_like(c2)).sqrt()

    def size(self, rho):
        v = self.m / rho
        return v if self.dim == 1 else v.sqrt() if self.dim == 2 else v ** (1.0 / 3.0)

    def cells(self, x, d, beta=0.0):
        """Cell index of every particle on the mesh of eq. (Dcell), and the mesh (cells per axis)."""
        top = torch.topk(d, 2).values
        dc = float(self.kh * (top[0] + top[1]) * (1.0 + beta) * (1.0 + 2.0 ** -20))
        c = torch.floor((x - x.min(0).values) * (1.0 / dc)).long()
        return c, (c.max(0).values + 1).tolist()

    def cell_order(self, x, d, beta=0.0):
        c, dims = self.cells(x, d, beta)
        lin = torch.zeros(len(c), dtype=torch.long, device=DEV)
        for a in reversed(range(self.dim)):
            lin = lin * dims[a] + c[:, a]
        return torch.sort(lin, stable=True).indices

    def pairs(self, x, d):
        """Interacting ordered pairs (i, j): r < kh (d_i + d_j)."""
        x, d = x.detach(), d.detach()
        c, dims = self.cells(x, d)
        dims = [k + 2 for k in dims]
        stride = [1]
        for k in dims[:-1]:
            stride.append(stride[-1] * k)
        lin = ((c + 1) * torch.tensor(stride, device=DEV)).sum(1)
        order = torch.sort(lin).indices
        keys = lin[order]
        I, J = [], []
        for off in itertools.product((-1, 0, 1), repeat=self.dim):
            want = lin + sum(o * s for o, s in zip(off, stride))
            lo, hi = torch.searchsorted(keys, want), torch.searchsorted(keys, want, right=True)
            cnt = hi - lo
            i = torch.repeat_interleave(torch.arange(len(lin), device=DEV), cnt)
            j = order[torch.arange(len(i), device=DEV) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt) + lo[i]]
            keep = ((x[j] - x[i]).square().sum(1) < (self.kh * (d[i] + d[j])).square()) & (i != j)
            I.append(i[keep])
            J.append(j[keep])
        return torch.cat(I), torch.cat(J)

    def dw(self, r, h):
        if self.q.kernel == "cubic":
            s = r / h
            norm = {1: 2.0 / 3.0, 2: 10.0 / (7.0 * math.pi), 3: 1.0 / math.pi}[self.dim] / h ** (self.dim + 1)
            return norm * torch.where(s < 1, s * (2.25 * s - 3), torch.where(s < 2, -0.75 * (2 - s) ** 2, torch.zeros_like(s)))
        H = self.q.kappa * h
        s = (r / H).clamp(max=1.0)
        if self.dim == 1:
            return 1.25 / H ** 2 * (-12 * s * (1 - s) ** 2)
        return {2: 7.0 / math.pi, 3: 21.0 / (2 * math.pi)}[self.dim] / H ** (self.dim + 1) * (-20 * s * (1 - s) ** 3)

    def evaluate(self, x, v, rho, E, d=None):
        """(a, drho, dE) at the given state; leaves d, P, c."""
        d = self.size(rho) if d is None else d
        P, c = self.eos(rho, E - 0.5 * v.square().sum(1))
        Z, V = rho * c, self.m / rho
        i, j = self.pairs(x, d)
        dx = x[j] - x[i]
        r = dx.square().sum(1).sqrt()
        e = dx / r[:, None]
        W = self.dw(r, 0.5 * self.q.eta * (d[i] + d[j]))
        vi, vj = (v[i] * e).sum(1), (v[j] * e).sum(1)
        Pi, Pj, wi, wj = P[i], P[j], vi, vj
        n = len(rho)
        add = lambda t: torch.zeros((n,) + t.shape[1:], dtype=t.dtype, device=DEV).index_add(0, i, t)  # noqa: E731
        if self.order == 2:
            f = -(V[j] * W)[:, None] * e
            gP = add(f * (Pj - Pi)[:, None])
            gv = add(f[:, None, :] * (v[j] - v[i])[:, :, None])
            mm = lambda a, b: torch.where((a > 0) & (b > 0), torch.minimum(a, b),  # noqa: E731
                                          torch.where((a < 0) & (b < 0), torch.maximum(a, b), torch.zeros_like(a)))
            slope = lambda k: r * torch.einsum("pa,pab,pb->p", e, gv[k], e)  # noqa: E731
            jP, jv = Pj - Pi, vj - vi
            Pi = P[i] + 0.5 * mm(r * (gP[i] * e).sum(1), jP)
            Pj = P[j] - 0.5 * mm(r * (gP[j] * e).sum(1), jP)
            wi, wj = vi + 0.5 * mm(slope(i), jv), vj - 0.5 * mm(slope(j), jv)
        Zi, Zj = Z[i], Z[j]
        if self.solver == "hll":
            Zi = Zj = torch.maximum(Zi, Zj)
        zs = Zi + Zj
        Ps = (Zj * Pi + Zi * Pj + Zi * Zj * (wi - wj)) / zs
        vs = (Zi * wi + Zj * wj + Pi - Pj) / zs
        F = 2 * V[i] * V[j] * Ps * W
        a = add(F[:, None] * e) / self.m[:, None]
        drho = 2 * rho * add(-V[j] * (vi - vs) * W)
        dE = add(F * vs) / self.m
        if self.unit is not None:
            K = self.K
            self.load = self.load + torch.bincount(self.unit[i], minlength=K).double()
            self.adj = self.adj | (torch.bincount(self.unit[i] * K + self.unit[j], minlength=K * K).view(K, K) > 0)
            dm = torch.full_like(d, -1.0).scatter_reduce(0, i, d[j], "amax")
            self.reach = torch.where(dm < 0, d, dm) + d
        self.d, self.P, self.c = d, P, c
        return a, drho, dE

    def step(self):
        if self.rates is None:
            self.rates = self.evaluate(self.x, self.v, self.rho, self.E)
        a, dr, de = self.rates
        with torch.no_grad():
            c = self.eos(self.rho, self.E - 0.5 * self.v.square().sum(1))[1]
            dt = float(self.q.cfl * (self.q.eta * self.size(self.rho) / (c + self.v.square().sum(1).sqrt())).min())
        h = 0.5 * dt
        v, rho, E = self.v + h * a, self.rho + h * dr, self.E + h * de
        self.x = self.x + dt * v
        self.rates = self.evaluate(self.x, v + h * a, rho + h * dr, E + h * de)
        a, dr, de = self.rates
        self.v, self.rho, self.E = v + h * a, rho + h * dr, E + h * de
        self.t += dt

    # ---- Voronoi work units
    def assign(self, gen):
        self.gen, self.K = gen, len(gen)
        x = self.x[:, : gen.shape[1]]
        self.unit = torch.cat([(x[k:k + 65536, None] - gen).square().sum(2).argmin(1) for k in range(0, len(x), 65536)])
        self.load = torch.zeros(self.K, dtype=torch.float64, device=DEV)
        self.adj = torch.zeros(self.K, self.K, dtype=torch.bool, device=DEV)

    def balance(self, theta=0.25, sigma=0.5, gamma_b=1.0, beta_sh=0.45):
        """Two-body and (2D) three-body displacement of the generators; returns the summed shift."""
        K, gd = self.gen.shape
        R = (1 + beta_sh) * self.kh * self.reach
        rmax = torch.zeros(K, dtype=torch.float64, device=DEV).scatter_reduce(0, self.unit, R, "amax").cpu().numpy()
        cnt = torch.bincount(self.unit, minlength=K).cpu().numpy()
        sums = torch.zeros(K, gd, dtype=torch.float64, device=DEV).index_add(0, self.unit, self.x[:, :gd]).cpu().numpy()
        L, adj, g = 0.5 * self.load.cpu().numpy(), self.adj.cpu().numpy(), self.gen.cpu().numpy()
        sig, new = (sigma if gd == 2 else 0.0), g.copy()
        rot = lambda t, w: np.array([w[0] * np.cos(t) - w[1] * np.sin(t), w[0] * np.sin(t) + w[1] * np.cos(t)])  # noqa: E731
        for k in range(K):
            near = [m for m in range(K) if m != k and adj[k, m]]
            two, three, dmax = np.zeros(gd), np.zeros(gd), max([max(rmax[k], rmax[m]) for m in near], default=0.0)
            for m in near:
                if L[k] + L[m] > 0:
                    w = g[k] - g[m]
                    two += max(rmax[k], rmax[m]) * (L[k] - L[m]) / (L[k] + L[m]) * w / np.linalg.norm(w)
            for a, b in itertools.combinations(near, 2):
                if sig == 0.0 or not adj[a, b] or not L[k] + L[a] + L[b] > 0:
                    continue
                u, w = g[a] - g[k], g[b] - g[k]
                cr = u[0] * w[1] - u[1] * w[0]
                if abs(cr) < 1e-12 * max(u @ u, w @ w):
                    continue
                o = g[k] + np.array([w[1] * (u @ u) - u[1] * (w @ w), u[0] * (w @ w) - w[0] * (u @ u)]) / (2 * cr)
                ck, turn = g[k] - o, 0.0
                for m in (a, b):
                    cm = g[m] - o
                    turn += np.sign(ck[0] * cm[1] - ck[1] * cm[0]) * math.pi / 3 * (L[m] - L[k]) / (L[k] + L[a] + L[b])
                three += rot(turn, ck) - ck
            length = np.linalg.norm(three)
            if length > dmax:
                three *= dmax / length
            rc = sums[k] / cnt[k] if cnt[k] else g[k]
            new[k] = (1 - theta) * (g[k] + gamma_b * ((1 - sig) * two + sig * three)) + theta * rc
        shift = float(np.linalg.norm(new - g, axis=1).sum())
        self.gen = _t(new)
        return shift

    def fields(self):
        out = {}
        a, dr, de = self.rates
        for k, ax in enumerate("xyz"[: self.dim]):
            out[ax], out["v" + ax], out["a" + ax] = self.x[:, k], self.v[:, k], a[:, k]
        out.update(rho=self.rho, E=self.E, drho=dr, dE=de, d=self.d, P=self.P, c=self.c, id=None)
        return out


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    with torch.no_grad():
        if case["kind"] == "ensemble":
            parts = []
            for q in _ensemble(case, seed):
                s = _Exact(q)
                for _ in range(case["steps"]):
                    s.step()
                parts.append(s.fields())
            return {k: None if v is None else torch.cat([p[k] for p in parts]) for k, v in parts[0].items()}
        q = _problem(case, seed)
        s = _Exact(q, case.get("order", 1), case.get("solver", "acoustic"))
        if case["kind"] == "balance":
            s.assign(_t(_disk_generators(case["K"])))
            a, dr, de = s.evaluate(s.x, s.v, s.rho, s.E)
            shift = s.balance()
            return dict(gen=s.gen, shift=np.array([shift]), offsets=None, unit=None,
                        rates=dict(ax=a[:, 0], ay=a[:, 1], az=a[:, 2], drho=dr, dE=de))
        return _exact_steps(case, q, s)


def _exact_steps(case, q, s):
    if case["units"]:
        s.assign(_t(synth.problem_generators(q)))
        s.permute(s.cell_order(s.x, s.size(s.rho), case["beta"]))       # the renumbering of build_cells
    for k in range(case["steps"]):
        s.step()
        if case["units"] and (k + 1) % case["n_upd"] == 0:
            s.balance()
            order = s.cell_order(s.x, s.d)
            s.assign(s.gen)
            s.permute(order)
    out = s.fields()
    if case["units"]:
        out.update(gen=s.gen, unit=None)
    if case["totals"]:
        mom = [(s.m * s.v[:, a]).sum() for a in range(s.dim)] + [torch.zeros((), dtype=torch.float64, device=DEV)] * (3 - s.dim)
        out["totals"] = torch.stack([s.m.sum()] + mom + [(s.m * s.E).sum()])[None]
    return out


def _exact_adjoint(case, seed):
    q = _problem(case, seed)
    f64 = dict(dtype=torch.float64, device=DEV)
    c0, gamma = torch.tensor(5300.0, **f64).requires_grad_(), torch.tensor(2.0, **f64).requires_grad_()
    s = _Exact(q, gamma=gamma, c0=c0)
    leaf = dict(pos=s.x, vel=s.v, rho=s.rho, E=s.E)
    for t in leaf.values():
        t.requires_grad_()
    weight = _loss_weight(s.v.detach()[:, 2])
    for _ in range(case["steps"]):
        s.step()
    (s.v[:, 2] * weight).sum().backward()
    leaf.update(c0=c0, gamma=gamma)
    return dict(pos=s.x.detach(), vel=s.v.detach(), rho=s.rho.detach(), E=s.E.detach(),
                grad={k: v.grad for k, v in leaf.items()})
