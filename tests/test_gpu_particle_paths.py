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
