"""Cases that stand for what a user has this framework do, and their FP64 restatement.

Three kinds of case, all driven through the public binding (``paper_2411_04703_gb300.api``):

* ``steps``: a loaded run is advanced some steps (``Sim.step``) and its fields E, B and current J
  are read into device tensors (``Sim.get_field``), as a program does between its diagnostics.  The
  workloads are the repository's own: the undulator in a periodic box (CIC or TSC), the plasma
  buncher in its moving window with absorbing sides (3-D and 2-D), the long undulator with absorbing
  faces, and the batched sweep.
* ``gradient``: checkpoints, steps and the reverse sweep (``Sim.checkpoint``, ``step``,
  ``backward``), one iteration of an optimiser over the undulator strength and the density profile.
* ``diagnostics``: the FP64 moments in both frames and the charge density of a loaded run.

``exact`` computes the small cases in 64 bits with plain torch, straight from the method's formulas
(no tiles, no sort, no windows, every ion a particle).
"""
from __future__ import annotations

import math

import torch

from paper_2411_04703_gb300 import api, workloads as W


# ----------------------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest run: thousands of electrons on a ragged grid, a few steps between looks at
        # the fields; launches and latency are all that counts
        dict(name="undulator tiny", kind="steps", physics="undulator", nx=20, ny=18, nz=44, n_beam=6000,
             order=1, steps=4),
        # the vacuum undulator at its own size, two sort periods per pass (L2-resident)
        dict(name="undulator 65k", kind="steps", physics="undulator", nx=32, ny=32, nz=64, n_beam=65536,
             order=1, steps=16),
        # second order, ragged grid, the undulator's cosh/sinh field and Vay's pusher
        dict(name="undulator tsc ragged", kind="steps", physics="undulator", nx=45, ny=39, nz=70,
             n_beam=300001, order=2, steps=8, vay=True, field_3d=True),
        # a quarter-size plasma buncher, the size of a parameter study
        dict(name="buncher small", kind="steps", physics="buncher", nx=64, ny=64, nz=128, n_beam=262144,
             order=2, ppc=222, steps=8),
        # the headline run: 61M plasma electrons at 8 per cell, 4.2M beam electrons, frozen ions
        dict(name="buncher", kind="steps", physics="buncher", nx=128, ny=128, nz=512, n_beam=4194304,
             order=2, ppc=222, steps=8),
        # the paper's own geometry, x-z
        dict(name="buncher 2d", kind="steps", physics="buncher", nx=1024, ny=1, nz=2048, n_beam=1048576,
             order=2, ppc=212, steps=8),
        # a dense bunch oscillating in a large grid with absorbing layers on every face
        dict(name="long undulator", kind="steps", physics="long", nx=256, ny=256, nz=1024,
             n_beam=33554432, order=2, steps=8),
        # the same bunch physics at the size of a test run, energy-conserving gather
        dict(name="long undulator small", kind="steps", physics="long", nx=63, ny=65, nz=200,
             n_beam=500000, order=2, steps=8, energy_gather=True),
        # 64 runs stacked in one context, plasma drifting 0.29 cells a step, a sort every 4 steps
        dict(name="sweep of 64", kind="steps", physics="sweep", runs=64, nx=64, ny=64, nz=128,
             n_beam=390000, order=2, ppc=122, steps=4, sort_every=4),
        # the differentiated run, twenty steps and their reverse sweep
        dict(name="gradient", kind="gradient", nx=64, ny=64, nz=256, n_beam=2097152, steps=20, every=10),
        # the smallest gradient, an optimiser's inner iteration on a toy grid
        dict(name="gradient tiny", kind="gradient", nx=16, ny=16, nz=32, n_beam=2000, steps=30, every=10),
        # what is read of a run between steps: both frames' moments and the charge density
        dict(name="diagnostics", kind="diagnostics", physics="buncher", nx=64, ny=64, nz=256,
             n_beam=2097152, order=2, ppc=222),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["undulator", "undulator", "buncher", "buncher", "buncher 2d", "long", "sweep", "gradient"])
    if kind == "undulator":
        return dict(kind="steps", physics="undulator", nx=_log_int(rng, 18, 96), ny=_log_int(rng, 18, 96),
                    nz=_log_int(rng, 44, 192), n_beam=_log_int(rng, 5000, 3000000), order=rng.choice([1, 2]),
                    steps=_log_int(rng, 2, 24), vay=rng.random() < 0.25, field_3d=rng.random() < 0.25,
                    energy_gather=rng.random() < 0.25)
    if kind == "buncher":
        return dict(kind="steps", physics="buncher", nx=_log_int(rng, 28, 128), ny=_log_int(rng, 26, 128),
                    nz=_log_int(rng, 64, 384), n_beam=_log_int(rng, 20000, 3000000), order=2,
                    ppc=rng.choice([122, 222, 212, 221]), steps=_log_int(rng, 3, 8))
    if kind == "buncher 2d":
        return dict(kind="steps", physics="buncher", nx=_log_int(rng, 64, 1000), ny=1, nz=_log_int(rng, 128, 2000),
                    n_beam=_log_int(rng, 20000, 1000000), order=2, ppc=rng.choice([212, 112, 313]),
                    steps=_log_int(rng, 3, 8))
    if kind == "long":
        return dict(kind="steps", physics="long", nx=_log_int(rng, 40, 200), ny=_log_int(rng, 40, 200),
                    nz=_log_int(rng, 100, 600), n_beam=_log_int(rng, 50000, 12000000), order=2,
                    steps=_log_int(rng, 3, 12))
    if kind == "sweep":
        return dict(kind="steps", physics="sweep", runs=_log_int(rng, 2, 16), nx=_log_int(rng, 24, 64),
                    ny=_log_int(rng, 24, 64), nz=8 * _log_int(rng, 5, 16), n_beam=_log_int(rng, 10000, 390000),
                    order=2, ppc=rng.choice([122, 222, 111]), steps=_log_int(rng, 2, 8),
                    sort_every=rng.choice([2, 3, 4]))
    return dict(kind="gradient", nx=_log_int(rng, 16, 56), ny=_log_int(rng, 16, 56), nz=_log_int(rng, 32, 200),
                n_beam=_log_int(rng, 2000, 1000000), steps=_log_int(rng, 8, 24), every=rng.choice([4, 6, 10]))


# ----------------------------------------------------------------------------- workloads

def _ppc(case):
    p = int(case.get("ppc", 0))
    return (p // 100, p // 10 % 10, p % 10)


def _workload(case, seed):
    """The repository's workload of a case at the case's size (a sweep: its Ensemble)."""
    grid = (case["nx"], case["ny"], case["nz"])
    n = case["n_beam"]
    if case["kind"] == "gradient":
        w = W.adjoint_workload(grid=grid, n_beam=n, steps=case["steps"], seed=seed)
        w.beam.sigma_r = min(w.beam.sigma_r, grid[0] / 8 * w.d[0])
        w.beam.sigma_z *= min(1.0, grid[2] / 64)
        return w
    physics = case["physics"]
    if physics == "undulator":
        w = W.vacuum_undulator(grid=grid, n_beam=n, seed=seed, order=case["order"])
        w.undulator.kind = 2 if case.get("field_3d") else 1
        return w
    if physics == "buncher":
        pml = 10 if min(grid[0], grid[1] if grid[1] > 1 else grid[0]) >= 40 else 4
        make = W.plasma_buncher_2d if grid[1] == 1 else W.plasma_buncher
        w = make(grid=grid, n_beam=n, seed=seed, pml=pml, ppc=_ppc(case))
        w.beam.sigma_z *= min(1.0, grid[2] / 256)     # the bunch stays inside a shorter window
        return w
    if physics == "long":
        # the bunch inside the field, as it is for most of the run (loaded by _bunch_in_field)
        w = W.long_undulator(grid=grid, n_beam=n, seed=seed, z_start=0.0)
        w.beam.sigma_r *= min(1.0, min(grid[0], grid[1]) / 64)
        return w
    # the lower half of the sweep's densities: above it the currents of electrons and ions cancel
    # to the rounding of 32 bits and two runs of one program differ in the percents
    e = W.batched_ensemble(runs=case["runs"], grid=grid, seed=seed, ppc=_ppc(case),
                           n_lab_cm3=(1e14, 1e15), n_beam_range=(n / 4, n * 2.5))
    e.base.beam.sigma_r *= min(1.0, min(grid[0], grid[1]) / 64)
    e.base.beam.sigma_z *= min(1.0, grid[2] / 128)
    return e


def _beam(w, seed):
    """The seeded lab-frame Gaussian beam of workloads.sample_beam, drawn on the GPU."""
    b = w.beam
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev).manual_seed(seed * 7919 + 13)
    r = torch.randn(6, b.n, generator=g, device=dev, dtype=torch.float64)
    x = r[:3] * torch.tensor([[b.sigma_r], [b.sigma_r], [b.sigma_z]], device=dev, dtype=torch.float64)
    u = torch.empty(3, b.n, device=dev, dtype=torch.float64)
    u[:2] = r[3:5] * (b.emit_n / b.sigma_r)
    gam = b.gamma * (1.0 + b.rel_spread * r[5])
    u[2] = (gam * gam - 1.0 - u[0] ** 2 - u[1] ** 2).sqrt()
    return x, u, torch.full((b.n,), b.weight, device=dev, dtype=torch.float64)


def _bunch_in_field(w, seed):
    """The long undulator's bunch some periods into the field, in the boosted frame at t' = 0: a
    Gaussian a twelfth of the grid long, every electron on its undulator orbit (zero transverse
    canonical momentum), so that it oscillates in place."""
    b, un = w.beam, w.undulator
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    g = torch.Generator(device=dev).manual_seed(seed * 7919 + 13)
    r = torch.randn(6, b.n, generator=g, device=dev, dtype=torch.float64)
    gR, bR = w.gamma_R, math.sqrt(1.0 - 1.0 / w.gamma_R ** 2)
    x = r[:3] * torch.tensor([[b.sigma_r], [b.sigma_r], [w.grid[2] * w.d[2] / 12]], device=dev, dtype=torch.float64)
    ph = 2 * math.pi / un.lambda_u * gR * (x[2] + b.origin[2] * w.d[2]) + un.phase
    u = torch.empty(3, b.n, device=dev, dtype=torch.float64)
    u[:2] = r[3:5] * (b.emit_n / b.sigma_r)
    u[0] += un.K * torch.sin(ph)
    up2 = u[0] ** 2 + u[1] ** 2
    gam = b.gamma * (1.0 + b.rel_spread * r[5])
    uz = (gam * gam - 1.0 - up2).sqrt()
    u[2] = gR * ((gam * gam / (gR * gR) - 1.0 - up2) / (uz + bR * gam))
    return x, u, torch.full((b.n,), b.weight, device=dev, dtype=torch.float64)


# ----------------------------------------------------------------------------- prepare and run

def prepare(case, seed):
    w = _workload(case, seed)
    if case.get("physics") == "sweep":
        tuning = {"tile": w.base.tile, "sort_every": case["sort_every"], "margin": 1}
        sim, ids = api.from_ensemble(w, tuning=tuning, beam=False)
        runs = [W.ensemble_run(w, r) for r in range(w.runs)]
        parts = [_beam(q, q.seed) for q in runs]
        x = torch.cat([p[0] for p in parts], dim=1)
        u = torch.cat([p[1] for p in parts], dim=1)
        wt = torch.cat([p[2] for p in parts])
        torch.cuda.synchronize()
        ids["beam"] = sim.load_species_batch(-1.0, 1.0, [q.beam.n for q in runs], x, u, wt,
                                             origin=w.base.beam.origin, match_undulator=True)
    elif case.get("physics") == "long":
        sim, ids = api.from_workload(w, beam=False)
        x, u, wt = _bunch_in_field(w, seed)
        torch.cuda.synchronize()
        ids["beam"] = sim.load_species(w.beam.q, w.beam.m, x, u, wt, frame=api.PIC_FRAME_BOOSTED,
                                       origin=w.beam.origin)
    else:
        arrays = _beam(w, seed)
        torch.cuda.synchronize()
        sim, ids = api.from_workload(w, beam_arrays=arrays)
    if case.get("vay"):
        sim.set_pusher(api.PIC_PUSHER_VAY)
    if case.get("energy_gather"):
        sim.set_gather(api.PIC_GATHER_ENERGY)
    state = {"case": case, "sim": sim, "ids": ids}
    shape = (3, sim.grid[2], sim.grid[1], sim.grid[0])
    if case["kind"] == "steps":
        for name in "EBJ":
            state[name] = torch.empty(shape, dtype=torch.float32, device="cuda")
    elif case["kind"] == "gradient":
        state["k"] = api.rrf_resonant_wavenumber(w)
    else:
        state["k"] = 2 * math.pi / (4 * w.d[2])
        state["k_lab"] = state["k"] / (w.gamma_R * (1 - math.sqrt(1 - 1 / w.gamma_R ** 2)
                                                    * math.sqrt(1 - 1 / w.beam.gamma ** 2)))
        state["rho"] = torch.empty(shape[1:], dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    return state


def run(state):
    case, sim, ids = state["case"], state["sim"], state["ids"]
    if case["kind"] == "gradient":
        sim.checkpoint(case["every"])
        sim.step(case["steps"])
        g = sim.backward(ids["beam"], state["k"])
        return {"loss": g["loss"], "dL_dK": g["dL_dK"], "dL_dprofile": g["dL_dprofile"].astype("float32")}
    if case["kind"] == "diagnostics":
        out = {"boosted": sim.get_moments(ids["beam"], api.PIC_FRAME_BOOSTED, state["k"]),
               "lab": sim.get_moments(ids["beam"], api.PIC_FRAME_LAB, state["k_lab"])}
        sim.get_field(api.PIC_RHO, out=state["rho"])
        out["rho"] = state["rho"]
        return out
    sim.step(case["steps"])
    for first, name in ((api.PIC_EX, "E"), (api.PIC_BX, "B"), (api.PIC_JX, "J")):
        for c in range(3):
            sim.get_field(first + c, out=state[name][c])
    return {name: state[name] for name in "EBJ"}


# ----------------------------------------------------------------------------- work

def _counts(case):
    """(cells, pushed particles, cells in absorbing layers) of a case."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    cells, n, pml = nx * ny * nz, case["n_beam"], 0
    if case["kind"] == "gradient":
        return cells, n + 4 * cells, 0
    physics = case["physics"]
    p = _ppc(case)
    ppc = p[0] * p[1] * p[2]
    if physics == "buncher":
        n += ppc * max(nx - 5, 0) * (ny - 5 if ny > 1 else 1) * (nz - 5)
        lay = 20 if min(nx, ny if ny > 1 else nx) >= 40 else 8
        pml = cells - (nx - lay) * ((ny - lay) if ny > 1 else 1) * nz
    elif physics == "long":
        pml = cells - (nx - 20) * (ny - 20) * (nz - 20)
    elif physics == "sweep":
        cells *= case["runs"]
        n = case["runs"] * n + ppc * cells
    return cells, n, pml


def work(case):
    cells, n, pml = _counts(case)
    if case["kind"] == "diagnostics":
        # the beam's records once, E and B once, every species' positions and weights for rho
        ions = n - case["n_beam"]
        return {"bytes": 32.0 * case["n_beam"] + 24.0 * cells + 20.0 * (n + ions) + 4.0 * cells,
                "flops": 200.0 * case["n_beam"] + 27 * 4.0 * (n + ions)}
    steps = case["steps"]
    nodes = 27 if case.get("order", 1) == 2 else 8
    push = 6 * nodes * 2 + 6 * nodes * 2 + 200
    # a step: each record (position and cell, momentum and weight) and E, B once in and once out;
    # the layers' auxiliaries (four a cell and layer) likewise; J once out at the end
    b = steps * (64.0 * n + 48.0 * cells + 32.0 * pml) + 36.0 * cells
    f = steps * (push * n + 60.0 * cells)
    if case["kind"] == "gradient":
        # the forward steps, the recomputed ones, and the sweep: the recorded state read, the
        # adjoints of records and fields read and written
        b = steps * (3 * 64.0 * n + 32.0 * n + 3 * 48.0 * cells + 24.0 * cells)
        f *= 4
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------- 64-bit restatement

def _shape(order, t):
    """Particle shape of order 0, 1 or 2 at distance t (cells)."""
    a = t.abs()
    if order == 0:
        return torch.ones_like(t)
    if order == 1:
        return (1.0 - a).clamp(min=0.0)
    return torch.where(a <= 0.5, 0.75 - a * a, 0.5 * (1.5 - a).clamp(min=0.0) ** 2)


class _Run:
    """One run of the method in 64 bits; positions in cells.  Every update makes new tensors, so
    that torch's autograd goes through it."""

    def __init__(self, w, gather=0, vay=False):
        self.w, self.gather, self.vay = w, gather, vay
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.n, self.d, self.dt = w.grid, w.d, w.dt
        self.per = [w.bc[k][0] == W.PERIODIC for k in range(3)]
        self.order = w.order
        self.gR = w.gamma_R
        self.bR = math.sqrt(1.0 - 1.0 / (w.gamma_R * w.gamma_R))
        nx, ny, nz = self.n
        self.E = [self._zeros() for _ in range(3)]
        self.B = [self._zeros() for _ in range(3)]
        self.J = [self._zeros() for _ in range(3)]
        self.K = torch.tensor(w.undulator.K if w.undulator else 0.0, dtype=torch.float64, device=self.dev)
        self.species = []
        self.step_no = 0
        self.coef = None
        if any(w.bc[k][f] == W.PML for k in range(3) for f in range(2)):
            self.coef = [[self._pml(k, 0), self._pml(k, 1)] for k in range(3)]
            self.psi = {}

    def _zeros(self):
        nx, ny, nz = self.n
        return torch.zeros(nz, ny, nx, dtype=torch.float64, device=self.dev)

    def _pml(self, k, half):
        n, L = self.n[k], float(self.w.pml)
        pos = torch.arange(n, dtype=torch.float64, device=self.dev) + 0.5 * half
        depth = torch.zeros_like(pos)
        if self.w.bc[k][0] == W.PML:
            depth = torch.where(pos < L, L - pos, depth)
        if self.w.bc[k][1] == W.PML:
            depth = torch.maximum(depth, (pos - ((n - 1) - L)).clamp(min=0.0))
        sig = 4.0 * -math.log(1e-8) / (2.0 * L * self.d[k]) * (depth / L) ** 3
        shape = [1, 1, 1]
        shape[2 - k] = n
        return torch.exp(-sig * self.dt * (0.5 if half else 1.0)).reshape(shape)

    # -- loading
    def add_beam(self, x, u, wt):
        """Lab particles at lab time 0: matched entry, Lorentz transform, drift to t' = 0."""
        w, d = self.w, self.d
        b = w.beam
        u = [u[0].clone(), u[1].clone(), u[2].clone()]
        un = w.undulator
        if un is not None and un.match:
            ku = 2 * math.pi / un.lambda_u
            g2 = 1.0 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2
            zl = x[2] + self.gR * b.origin[2] * d[2]
            ch = torch.cosh(ku * (x[1] + b.origin[1] * d[1] - 0.5 * self.n[1] * d[1])) if un.kind == 2 else 1.0
            u[0] = u[0] + un.K * ch * torch.sin(ku * zl + un.phase)
            u[2] = (g2 - 1.0 - u[0] ** 2 - u[1] ** 2).sqrt()
        up2 = u[0] ** 2 + u[1] ** 2
        g = (1.0 + up2 + u[2] ** 2).sqrt()
        ig2 = 1.0 / (self.gR * self.gR)
        uz = self.gR * ((g * g * ig2 - 1.0 - up2) / (u[2] + self.bR * g))
        gp = self.gR * ((1.0 + up2 + u[2] ** 2 * ig2) / (g + self.bR * u[2]))
        drift = self.gR * self.bR * x[2] / gp
        X = [(x[0] + drift * u[0]) / d[0] + b.origin[0], (x[1] + drift * u[1]) / d[1] + b.origin[1],
             (self.gR * x[2] + drift * uz) / d[2] + b.origin[2]]
        self._add(torch.stack(X, 1), torch.stack([u[0], u[1], uz], 1), wt, -1.0, 1.0, False)

    def add_plasma(self, profile=None):
        """The lab-static lattice: electrons and immobile ions on the same points."""
        p, n, d = self.w.plasma, self.n, self.d
        lo, hi = (1, 2) if self.order == 1 else (2, 3)
        if self.per[2]:
            m0, m1 = 0, p.ppc[2] * n[2] - 1
        else:
            m0 = math.ceil(p.ppc[2] * lo - 0.5)
            m1 = math.ceil(p.ppc[2] * (n[2] - hi) - 0.5) - 1
        f = dict(dtype=torch.float64, device=self.dev)
        z = (torch.arange(m0, m1 + 1, **f) + 0.5) / p.ppc[2]
        ax = []
        for k in range(2):
            a, e = p.xrange[2 * k], p.xrange[2 * k + 1]
            ax.append(a + (torch.arange((e - a) * p.ppc[k], **f) + 0.5) / p.ppc[k])
        zn = torch.tensor(p.z_nodes, **f)
        dn = torch.tensor(p.n_nodes, **f) if profile is None else profile
        zl = self.gR * z * d[2]
        i = (torch.searchsorted(zn, zl) - 1).clamp(0, len(zn) - 2)
        r = (zl - zn[i]) / (zn[i + 1] - zn[i])
        dens = self.gR * (dn[i] + r * (dn[i + 1] - dn[i])) * (d[0] * d[1] * d[2]) / (p.ppc[0] * p.ppc[1] * p.ppc[2])
        Z, Y, X = torch.meshgrid(z, ax[1], ax[0], indexing="ij")
        x = torch.stack([X.reshape(-1), Y.reshape(-1), Z.reshape(-1)], 1)
        wt = dens[:, None].expand(-1, len(ax[0]) * len(ax[1])).reshape(-1)
        u = torch.zeros_like(x)
        u[:, 2] = -self.gR * self.bR
        self._add(x, u, wt, -1.0, 1.0, False)
        self._add(x, u, wt, 1.0, 1836.15267343, True)

    def _add(self, x, u, wt, q, m, frozen):
        x, keep = self._wrap(x)
        self.species.append(dict(x=x[keep], u=u[keep], w=wt[keep], q=q, m=m, frozen=frozen))

    def _wrap(self, x):
        lo, hi = (1, 2) if self.order == 1 else (2, 3)
        keep = torch.ones(len(x), dtype=torch.bool, device=x.device)
        cols = []
        for k in range(3):
            c = x[:, k]
            if self.per[k]:
                c = c - self.n[k] * torch.floor(c.detach() / self.n[k])
            else:
                keep &= (c >= lo) & (torch.floor(c) <= self.n[k] - 1 - hi)
            cols.append(c)
        return torch.stack(cols, 1), keep

    # -- one dimension's window: node indices (wrapped or -1) and weights
    def _nodes(self, k, first, count):
        i = first[:, None] + torch.arange(count, device=first.device)
        if self.per[k]:
            return i % self.n[k], None
        ok = (i >= 0) & (i < self.n[k])
        return i.clamp(0, self.n[k] - 1), ok

    def _interp(self, F, x, stag):
        idx, wts = [], []
        for k in range(3):
            o = self.order - (1 if self.gather and stag[k] else 0)
            t = x[:, k] - (0.5 if stag[k] else 0.0)
            first = (torch.floor(t) if o == 1 else torch.floor(t + 0.5) - (1 if o == 2 else 0)).detach().long()
            wt = _shape(o, t[:, None] - (first[:, None] + torch.arange(o + 1, device=x.device)))
            i, ok = self._nodes(k, first, o + 1)
            wts.append(wt if ok is None else wt * ok)
            idx.append(i)
        nx, ny, _ = self.n
        flat = (idx[2][:, :, None, None] * ny + idx[1][:, None, :, None]) * nx + idx[0][:, None, None, :]
        return torch.einsum("nkji,nk,nj,ni->n", F.reshape(-1)[flat], wts[2], wts[1], wts[0])

    def _external(self, x):
        un = self.w.undulator
        if un is None:
            return 0.0, 0.0
        ku = 2 * math.pi / un.lambda_u
        zl = self.gR * (x[:, 2] * self.d[2] + self.bR * self.step_no * self.dt)
        f = 1.0
        if math.isfinite(un.z_start) and un.ramp >= 0.0:
            f = ((zl - un.z_start) / un.ramp).clamp(0.0, 1.0)
        B0 = self.K * ku * f
        ph = ku * zl + un.phase
        By, Bz = self.gR * B0 * torch.cos(ph), 0.0
        if un.kind == 2:
            ky = ku * (x[:, 1] - 0.5 * self.n[1]) * self.d[1]
            Bz = -B0 * torch.sinh(ky) * torch.sin(ph)
            By = By * torch.cosh(ky)
        return By, Bz

    def _push(self, s, x, u):
        F = [self._interp(self.E[c], x, [c == k for k in range(3)]) for c in range(3)]
        G = [self._interp(self.B[c], x, [c != k for k in range(3)]) for c in range(3)]
        By, Bz = self._external(x)
        F[0], G[1], G[2] = F[0] - self.bR * By, G[1] + By, G[2] + Bz
        E, B = torch.stack(F, 1), torch.stack(G, 1)
        h = 0.5 * s["q"] / s["m"] * self.dt
        gam = lambda v: (1.0 + (v * v).sum(1, keepdim=True)).sqrt()  # noqa: E731
        cross = lambda a, b: torch.linalg.cross(a, b, dim=1)  # noqa: E731
        if self.vay:
            up = u + h * (2.0 * E + cross(u / gam(u), B))
            tau = h * B
            us = (up * tau).sum(1, keepdim=True)
            t2 = (tau * tau).sum(1, keepdim=True)
            sg = gam(up) ** 2 - t2
            g1 = (0.5 * (sg + (sg * sg + 4.0 * (t2 + us * us)).sqrt())).sqrt()
            t = tau / g1
            return (up + (up * t).sum(1, keepdim=True) * t + cross(up, t)) / (1.0 + (t * t).sum(1, keepdim=True))
        um = u + h * E
        t = h * B / gam(um)
        up = um + cross(um, t)
        return um + cross(up, 2.0 * t / (1.0 + (t * t).sum(1, keepdim=True))) + h * E

    def _deposit(self, x, dx, qw):
        """Esirkepov's current of a move by dx (cells) from x, on a window wide enough for it."""
        L = self.order + 3
        S0, DS, idx, oks = [], [], [], []
        for k in range(3):
            first = (torch.floor(x[:, k] + (0.5 if self.order == 2 else 0.0)) - self.order).detach().long()
            nodes = first[:, None] + torch.arange(L, device=x.device)
            a = _shape(self.order, x[:, k, None] - nodes)
            S0.append(a)
            DS.append(_shape(self.order, (x[:, k] + dx[:, k])[:, None] - nodes) - a)
            i, ok = self._nodes(k, first, L)
            idx.append(i)
            oks.append(ok)
        nx, ny, _ = self.n
        flat = ((idx[2][:, :, None, None] * ny + idx[1][:, None, :, None]) * nx + idx[0][:, None, None, :])
        ok = None
        for k, o in enumerate(oks):
            if o is not None:
                o = o.reshape([len(x)] + [L if j == 2 - k else 1 for j in range(3)])
                ok = o if ok is None else ok & o
        V = self.d[0] * self.d[1] * self.d[2]
        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            T = (S0[a][:, :, None] * S0[b][:, None, :] + 0.5 * DS[a][:, :, None] * S0[b][:, None, :]
                 + 0.5 * S0[a][:, :, None] * DS[b][:, None, :] + DS[a][:, :, None] * DS[b][:, None, :] / 3.0)
            P = DS[c].cumsum(1) * (-qw * self.d[c] / (self.dt * V))[:, None]
            val = torch.einsum("np,nqr->npqr", P, T).permute(
                [0] + [1 + [c, a, b].index(k) for k in (2, 1, 0)])
            if ok is not None:
                val = val * ok
            self.J[c] = self.J[c].reshape(-1).index_add(0, flat.reshape(-1), val.reshape(-1)).reshape(self.J[c].shape)

    def step(self, chunk=1 << 20):
        self.J = [self._zeros() for _ in range(3)]
        for s in self.species:
            xs, us, keeps = [], [], []
            for lo in range(0, len(s["x"]), chunk):
                x, u, wt = s["x"][lo:lo + chunk], s["u"][lo:lo + chunk], s["w"][lo:lo + chunk]
                if not s["frozen"]:
                    u = self._push(s, x, u)
                g = (1.0 + (u * u).sum(1, keepdim=True)).sqrt()
                dx = u / g * torch.tensor([self.dt / v for v in self.d], dtype=torch.float64, device=x.device)
                x1, keep = self._wrap(x + dx)
                self._deposit(x, dx, s["q"] * torch.where(keep, wt, torch.zeros_like(wt)))
                xs.append(x1)
                us.append(u)
                keeps.append(keep)
            if xs:
                keep = torch.cat(keeps)
                x, u = torch.cat(xs), torch.cat(us)
                s["x"], s["u"], s["w"] = (x, u, s["w"]) if bool(keep.all()) else (x[keep], u[keep], s["w"][keep])
        self._faraday(0.5 * self.dt)
        self._ampere()
        self._faraday(0.5 * self.dt)
        self.step_no += 1

    def _diff(self, F, k, way, key, half):
        """Forward (way = 1) or backward difference along dim k, stretched in the layers."""
        ax = 2 - k
        G = torch.roll(F, -way, ax)
        if not self.per[k]:
            edge = [slice(None)] * 3
            edge[ax] = -1 if way == 1 else 0
            mask = torch.ones_like(F)
            mask[tuple(edge)] = 0.0
            G = G * mask
        D = way * (G - F) / self.d[k]
        if self.coef is None:
            return D
        b = self.coef[k][half]
        self.psi[key] = b * self.psi.get(key, 0.0) + (b - 1.0) * D
        return D + self.psi[key]

    def _curl(self, F, way, tag, half):
        D = lambda c, k: self._diff(F[c], k, way, (tag, c, k), half)  # noqa: E731
        return [D(2, 1) - D(1, 2), D(0, 2) - D(2, 0), D(1, 0) - D(0, 1)]

    def _faraday(self, h):
        c = self._curl(self.E, 1, "B", 1)
        self.B = [b - h * v for b, v in zip(self.B, c)]

    def _ampere(self):
        c = self._curl(self.B, -1, "E", 0)
        self.E = [e + self.dt * (v - j) for e, v, j in zip(self.E, c, self.J)]

    def rho(self):
        out = self._zeros().reshape(-1)
        V = self.d[0] * self.d[1] * self.d[2]
        nx, ny, _ = self.n
        for s in self.species:
            for lo in range(0, len(s["x"]), 1 << 21):
                x, wt = s["x"][lo:lo + (1 << 21)], s["w"][lo:lo + (1 << 21)]
                idx, wts = [], []
                for k in range(3):
                    first = (torch.floor(x[:, k]) if self.order == 1 else torch.floor(x[:, k] + 0.5) - 1).long()
                    v = _shape(self.order, x[:, k, None] - (first[:, None] + torch.arange(self.order + 1, device=x.device)))
                    i, ok = self._nodes(k, first, self.order + 1)
                    idx.append(i)
                    wts.append(v if ok is None else v * ok)
                flat = (idx[2][:, :, None, None] * ny + idx[1][:, None, :, None]) * nx + idx[0][:, None, None, :]
                val = torch.einsum("nk,nj,ni,n->nkji", wts[2], wts[1], wts[0], s["q"] * wt / V)
                out.index_add_(0, flat.reshape(-1), val.reshape(-1))
        return out.reshape(self._zeros().shape)


def _quiet(w, steps):
    """Whether no window shift and no plasma plane falls into the first steps of a run."""
    if not w.moving_window:
        return True
    if math.floor(w.window_v * steps * w.dt / w.d[2]) > 0:
        return False
    hi = 2 if w.order == 1 else 3
    bR = math.sqrt(1.0 - 1.0 / w.gamma_R ** 2)
    plane = lambda n: math.ceil(w.plasma.ppc[2] * (w.grid[2] - hi + bR * n * w.dt / w.d[2]) - 0.5)  # noqa: E731
    return plane(steps) == plane(0)


def exact(case, seed):
    cells, n, _ = _counts(case)
    if case["kind"] == "gradient":
        if n * case["steps"] > 3e6:
            return None
        w = _workload(case, seed)
        s = _Run(w)
        s.K.requires_grad_(True)
        profile = torch.tensor(w.plasma.n_nodes, dtype=torch.float64, device=s.dev, requires_grad=True)
        s.add_plasma(profile)
        s.add_beam(*_beam(w, seed))
        for _ in range(case["steps"]):
            s.step()
        b = s.species[-1]
        un = w.undulator
        gB = w.beam.gamma
        bz1 = (1.0 + 0.5 * un.K ** 2) / (2.0 * gB * gB)        # 1 - beta_z of the beam
        k = 4 * math.pi * gB * gB / (un.lambda_u * (1.0 + 0.5 * un.K ** 2))
        k *= s.gR * (1.0 / (s.gR ** 2 * (1.0 + s.bR)) + s.bR * bz1)
        ph = k * b["x"][:, 2] * w.d[2]
        re, im = (b["w"] * torch.cos(ph)).sum(), (b["w"] * torch.sin(ph)).sum()
        loss = (re * re + im * im).sqrt() / b["w"].sum()
        _, dP = torch.autograd.grad(loss, [s.K, profile])
        # the loss and dL/dK are single numbers whose 32-bit rounding varies fifty-fold between
        # seeds (5e-7 to 4e-5 of dL/dK): their distance from this value measures chance
        return {"loss": None, "dL_dK": None, "dL_dprofile": dP.detach().cpu().numpy()}
    with torch.no_grad():
        if case["kind"] == "diagnostics":
            w = _workload(case, seed)
            s = _Run(w)
            s.add_plasma()
            s.add_beam(*_beam(w, seed))
            return {"boosted": None, "lab": None, "rho": s.rho()}
        if (2 * n - case["n_beam"]) * case["steps"] > 6e7:
            return None
        if case["physics"] == "sweep":
            e = _workload(case, seed)
            runs = [W.ensemble_run(e, r) for r in range(e.runs)]
        else:
            runs = [_workload(case, seed)]
        out = {"E": [], "B": [], "J": []}
        for w in runs:
            if not _quiet(w, case["steps"]):
                return None
            s = _Run(w, gather=int(bool(case.get("energy_gather"))), vay=bool(case.get("vay")))
            if w.plasma is not None:
                s.add_plasma()
            if case["physics"] == "long":
                x, u, wt = _bunch_in_field(w, w.seed)
                at = [x[k] / w.d[k] + w.beam.origin[k] for k in range(3)]
                s._add(torch.stack(at, 1), u.T, wt, -1.0, 1.0, False)
            else:
                s.add_beam(*_beam(w, w.seed))
            for _ in range(case["steps"]):
                s.step()
            for name, F in (("E", s.E), ("B", s.B), ("J", s.J)):
                out[name].append(torch.stack(F))
        return {name: torch.cat(v, dim=1) for name, v in out.items()}
