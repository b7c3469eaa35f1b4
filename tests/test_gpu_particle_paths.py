"""The particle kernel's paths against the FP64 oracle, one step from an identical state, at the
sizes where each can go wrong.  Tolerance: the repository's bar of one step, 1e-5 of the largest
value per component (FP32 gather, push and deposit round at 6e-8 each, a few tens of them).
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


def _one_step(w, sim, ids, seed, gather=0):
    rng = np.random.default_rng(seed)
    for c in range(6):
        sim.set_field(c, (1e-3 * rng.standard_normal((w.grid[2], w.grid[1], w.grid[0]))).astype(np.float32))
    o, oid = parity.oracle_from_gpu(w, sim, ids)
    if gather:
        o.set_gather(1)
    sim.step(1)
    sim.sync()
    o.step(1)
    for name in ids:
        r = parity.compare_species(w, sim, ids[name], o, oid[name])
        assert r["only_gpu"] == 0 and r["only_oracle"] == 0 and r["cell_mismatch"] == 0, (name, r)
        assert r["u_rel_err"] < TOL_STEP and r["pos_abs_err"] < 1e-5, (name, r)
    f = parity.compare_fields(sim, o)
    assert max(f.values()) < TOL_STEP, f


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("grid", [(7, 5, 9), (9, 1, 17), (2, 3, 8), (20, 18, 44)])
@pytest.mark.parametrize("gather", [0, 1])
def test_few_particles_per_tile(grid, order, gather):
    # tiles with fewer than 32 particles take the global-memory path; short periodic dims wrap
    # once or several times inside one window
    w = W.vacuum_undulator(grid=grid, n_beam=25, seed=3, order=order)
    sim, ids = api.from_workload(w)
    sim.set_gather(gather)
    _one_step(w, sim, ids, 5, gather)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("steps", [3, 7, 14])
def test_particles_drifted_from_their_tiles(order, steps):
    # the bunch drifts 0.23 cells a step: inside the margin, partly and wholly beyond it, since the
    # last sort
    w = W.mini_vacuum(order=order)
    sim, ids = api.from_workload(w, tuning={"tile": (8, 8, 8), "sort_every": 32, "margin": 1})
    sim.step(steps)
    _one_step(w, sim, ids, 7)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("gather", [0, 1])
@pytest.mark.parametrize("n", [33, 700, 9000])
def test_hot_particles_cross_nodes(order, gather, n):
    # random relativistic momenta: moves of up to 0.28 cells along each dim, so that the nearest node
    # changes along none, one, two or all dims, in both directions
    w = W.vacuum_undulator(grid=(20, 10, 18), n_beam=n, seed=3, order=order)
    w.undulator = None
    X, U, Wt = W.sample_uniform_particles(w.grid, n, seed=21 + n, umax=4.0)
    if n == 33:
        X = 8.0 + 1.5 * (X / np.array(w.grid))      # one tile just above the sparse limit
    sim, ids = api.from_workload(w, beam=False)
    ids["beam"] = sim.load_species(-1.0, 1.0, X.T * np.array(w.d)[:, None], U.T, Wt * 1e-3,
                                   frame=api.PIC_FRAME_BOOSTED)
    sim.set_gather(gather)
    _one_step(w, sim, ids, 9, gather)


@pytest.mark.parametrize("tile", [(8, 8, 8), (1, 16, 5), (16, 3, 4), (5, 5, 5), (10, 8, 8), (2, 1, 2)])
@pytest.mark.parametrize("margin", [0, 1, 2])
def test_tile_shapes_and_margins(tile, margin):
    # regions of other shapes (one to four CTAs per SM) and drift margins, after five steps of drift
    w = W.mini_dense_bunch(order=2, n_beam=20000)
    try:
        sim, ids = api.from_workload(w, tuning={"tile": tile, "sort_every": 8, "margin": margin})
    except api.PicError:
        pytest.skip("the region of this tile exceeds shared memory")
    sim.step(5)
    _one_step(w, sim, ids, 13)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("tile", [(8, 8, 8), (5, 4, 6)])
def test_frozen_particle_species(order, tile):
    # a frozen species held as particles (its own kernel) beside a mobile one
    w = W.vacuum_undulator(grid=(20, 10, 18), n_beam=3000, seed=3, order=order)
    w.undulator = None
    sim, ids = api.from_workload(w, beam=False, tuning={"tile": tile, "sort_every": 4, "margin": 1})
    for name, q, m, seed, frozen in (("plasma_i", 1.0, 1836.15267343, 31, True), ("beam", -1.0, 1.0, 32, False)):
        X, U, Wt = W.sample_uniform_particles(w.grid, 9000, seed=seed, umax=3.0)
        ids[name] = sim.load_species(q, m, X.T * np.array(w.d)[:, None], U.T, Wt * 1e-3,
                                     frame=api.PIC_FRAME_BOOSTED, frozen=frozen)
    sim.step(2)
    _one_step(w, sim, ids, 11)
