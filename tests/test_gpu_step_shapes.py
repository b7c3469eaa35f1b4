"""The field updates' launch shapes and the end of a step against the FP64 oracle.  Tolerance: the
repository's bar of one step, 1e-5 of the largest value per component, times the steps taken.
"""
import numpy as np
import pytest

import oracle
from paper_2411_04703_gb300 import api, workloads as W

import parity

pytestmark = pytest.mark.gpu

TOL_STEP = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    oracle.build()


# walks of 1 cell (with 1, 2, 3 and more rows of y, ragged in every dim), 2, 4 and 8 cells, the last
# walk of a column cut short
@pytest.mark.parametrize("grid", [(9, 1, 30), (300, 1, 21), (40, 2, 33), (5, 3, 70), (33, 7, 41),
                                  (33, 64, 233), (33, 64, 461), (33, 64, 919)])
@pytest.mark.parametrize("layers", [False, True])
def test_field_update_shapes(grid, layers):
    d, dt = (0.5, 0.6, 0.55), 0.27
    face = [(W.PML, W.PML) if layers and n >= 20 else (W.PERIODIC, W.PERIODIC) for n in grid]
    sim = api.Sim(grid, d, dt, 1.0, bc=face, pml=6 if layers else 0)
    o = oracle.Sim(grid, d, dt, 1.0, bc=face, pml=6 if layers else 0)
    rng = np.random.default_rng(sum(grid))
    for c in range(6):
        f = rng.standard_normal((grid[2], grid[1], grid[0])).astype(np.float32)
        sim.set_field(c, f)
        o.set_field(c, f.astype(np.float64))
    steps = 2                                   # the second meets the layers' psi of the first
    sim.step(steps)
    sim.sync()
    for _ in range(steps):
        o.fdtd()
    f = parity.compare_fields(sim, o, range(6))
    assert max(f.values()) < steps * TOL_STEP, f


@pytest.mark.parametrize("n_species", [1, 3, 8])
def test_step_end_serves_every_species(n_species):
    # each species has its own bound on a step's displacement, its own counters and the common clock
    w = W.vacuum_undulator(grid=(20, 10, 18), n_beam=900, seed=3, order=2)
    sim, _ = api.from_workload(w, beam=False)
    o, oid = parity.oracle_from_gpu(w, sim, {})
    ids = []
    for s in range(n_species):
        X, U, Wt = W.sample_uniform_particles(w.grid, 900, seed=50 + s, umax=0.02 * 2.0 ** s)
        ids.append(sim.load_species(-1.0, 1.0, X.T * np.array(w.d)[:, None], U.T, Wt * 1e-3, frame=api.PIC_FRAME_BOOSTED))
        P = sim.get_particles(ids[s])
        oid[s] = o.add_species(-1.0, 1.0, capacity=1024)
        o.set_state(oid[s], P["cell"].astype(np.float64) + P["off"].astype(np.float64), P["u"].astype(np.float64),
                    P["w"].astype(np.float64), P["id"])
    steps = 3
    sim.step(steps)
    sim.sync()
    o.step(steps)
    assert sim.get_time()[0] == steps
    w.beam.q, w.beam.m = -1.0, 1.0
    for s in range(n_species):
        r = parity.compare_species(w, sim, ids[s], o, oid[s])
        assert r["only_gpu"] == 0 and r["only_oracle"] == 0, (s, r)
        assert r["u_rel_err"] < steps * TOL_STEP and r["pos_abs_err"] < steps * 1e-5, (s, r)
    f = parity.compare_fields(sim, o)
    assert max(f.values()) < steps * TOL_STEP, f


# One particle, a cold pair, a hot cloud: the two passes' shift about the mean particle.  FP64 on the
# same records: 1e-9 of a value; a spread also within 1e-7 of the largest coordinate, ten times the root
# of FP64 rounding (a single particle has none).
@pytest.mark.parametrize("n, umax", [(1, 0.5), (2, 0.0), (3000, 4.0)])
@pytest.mark.parametrize("frame, oframe", [(api.PIC_FRAME_LAB, 1), (api.PIC_FRAME_BOOSTED, 0)])
def test_moments_in_two_passes(n, umax, frame, oframe):
    w = W.vacuum_undulator(grid=(20, 10, 18), n_beam=n, seed=3, order=2)
    sim, _ = api.from_workload(w, beam=False)
    o, _ = parity.oracle_from_gpu(w, sim, {})
    X, U, Wt = W.sample_uniform_particles(w.grid, n, seed=70 + n, umax=umax)
    sid = sim.load_species(-1.0, 1.0, X.T * np.array(w.d)[:, None], U.T, Wt, frame=api.PIC_FRAME_BOOSTED)
    P = sim.get_particles(sid)
    s = o.add_species(-1.0, 1.0, capacity=max(n, 1))
    o.set_state(s, P["cell"].astype(np.float64) + P["off"].astype(np.float64), P["u"].astype(np.float64),
                P["w"].astype(np.float64), P["id"])
    g, r = sim.get_moments(sid, frame, k_bunch=3.0), o.moments(s, frame=oframe, k=3.0)
    scale = max(abs(r[k]) for k in ("mean_x", "mean_y", "mean_z", "mean_gamma"))
    for k in ("count", "mean_x", "mean_y", "mean_z", "mean_uz", "mean_gamma", "bunching", "kinetic_energy", "mean_t"):
        assert g[k] == pytest.approx(r[k], rel=1e-9, abs=1e-12), (k, g[k], r[k])
    for k in ("rms_x", "rms_y", "rms_z", "rel_energy_spread", "emit_nx", "emit_ny"):
        assert g[k] == pytest.approx(r[k], rel=1e-9, abs=1e-7 * scale), (k, g[k], r[k])


# A small energy spread beside a large transverse momentum: the Lorentz factor of the mean momentum is far
# from the mean one.  Bound: a record's Lorentz factor in its frame is some eight FP64 roundings, and the
# spread about their mean no further off than they are, 8 x 1.1e-16 of the mean, times ten.
@pytest.mark.parametrize("frame", [api.PIC_FRAME_LAB, api.PIC_FRAME_BOOSTED])
@pytest.mark.parametrize("ux, uz", [(1.0, 3.0), (100.0, 0.5), (0.5, -20.0)])
def test_energy_spread_beside_a_transverse_oscillation(frame, ux, uz):
    w = W.vacuum_undulator(grid=(20, 10, 18), n_beam=4, seed=3, order=2)
    sim, _ = api.from_workload(w, beam=False)
    n, rng = 20000, np.random.default_rng(5)
    X = rng.uniform(4.0, 9.0, (3, n)) * np.array(w.d)[:, None]
    U = np.stack([ux * np.where(np.arange(n) % 2, 1.0, -1.0), np.zeros(n), uz * (1.0 + 1e-6 * rng.standard_normal(n))])
    sid = sim.load_species(-1.0, 1.0, X, U, np.ones(n), frame=api.PIC_FRAME_BOOSTED)
    u = sim.get_particles(sid)["u"].astype(np.longdouble)
    g = np.sqrt(1 + (u ** 2).sum(1))
    if frame == api.PIC_FRAME_LAB:
        gR = np.longdouble(w.gamma_R)
        g = gR * (g + np.sqrt(1 - 1 / gR ** 2) * u[:, 2])
    spread = float(np.sqrt(((g - g.mean()) ** 2).mean()) / g.mean())
    m = sim.get_moments(sid, frame, k_bunch=3.0)
    assert m["mean_gamma"] == pytest.approx(float(g.mean()), rel=1e-13)
    assert abs(m["rel_energy_spread"] - spread) < 80 * 1.1e-16, (m["rel_energy_spread"], spread)
