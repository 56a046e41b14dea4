"""Particles that leave through absorbing and source walls, which the plain push settles in its
common path: few cells, fast particles, several of a quad at once, beside candidates and
empty slots, and more cells than the settled words can tell apart; against the oracle."""
import dataclasses

import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import assert_same_clocks, by_id, particle_errors, requires_gpu, run_gpu, run_oracle

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ncells,ppc,dt", [(1, 300, 0.05), (3, 200, 0.4), (17, 50, 0.4), (40, 33, 1.0)])
@pytest.mark.parametrize("bc,nstep", [(W.BC_ABSORB, 1), (W.BC_ABSORB, 3), (W.BC_SOURCE, 1)])
def test_walls_match_the_oracle(bc, nstep, ncells, ppc, dt):
    phys = dataclasses.replace(W.bounded_small(ncells=ncells, ppc=ppc, seed=9, nu=0.2, ion_nstep=nstep),
                               dt=dt, bc=bc)
    loads = W.initial_load(phys, seed=9)
    g, gm = run_gpu(phys, loads, 30, capi.FP64, sort_interval=7)
    o, om = run_oracle(phys, loads, 30)
    for k in ("live", "wall_count", "collisions"):
        np.testing.assert_array_equal(gm[k], om[k], err_msg=k)
    np.testing.assert_allclose(gm["wall_energy"], om["wall_energy"], rtol=1e-12)
    assert_same_clocks(g, o)
    for ex, ev in particle_errors(phys, g, o):
        assert ex < 1e-12 and ev < 1e-12


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
@pytest.mark.parametrize("ncells", [(1 << 21) - 1, 1 << 21, (1 << 21) + 1, (1 << 22) + 1])
def test_walls_of_many_cells(ncells, precision):
    """Particles in the first and last cells, at speeds up to and past the cells that a word can
    tell apart: counts and what stays, against the same sum in the form's precision and Python
    integers."""
    j, u = np.meshgrid([0, 1, 5, ncells // 2, ncells - 2, ncells - 1],
                       [0.0, 0.5, 1.25, 3.0, 2.0 ** 20 - 1, 2.0 ** 20, 2.0 ** 21, 2.0 ** 22])
    j, u = np.repeat(j.ravel(), 2).astype(np.int64), np.repeat(u.ravel(), 2)
    u[1::2] *= -1.0
    n = len(j)
    off, zero = np.full(n, 0.25), np.zeros(n)
    phys = W.Physics(ncells=ncells, dx=1.0, dt=1.0, processes=[], bc=W.BC_ABSORB, field=W.FIELD_NONE,
                     species=[W.Species("n", 0.0, 1.0, 1.0, 0.0, 1)])
    sim = capi.Sim(phys, precision=precision, sort_interval=0, capacity=[[n]])
    sim.load(0, 0, W.Load(j.astype(np.int32), off, u, zero, zero.copy(), np.arange(n, dtype=np.uint32)))
    sim.step(1)
    m, p = sim.moments(0), by_id(sim.particles(0, 0))
    sim.close()
    t = np.float32 if precision == capi.FP32 else np.float64
    f = t(0.25) + u.astype(t)
    x = j + np.floor(f).astype(np.int64)
    stay = (x >= 0) & (x < ncells)
    np.testing.assert_array_equal(m["wall_count"][0], [(x < 0).sum(), (x >= ncells).sum()])
    np.testing.assert_array_equal(p["id"], np.nonzero(stay)[0])
    np.testing.assert_array_equal(p["cell"], x[stay])
    np.testing.assert_array_equal(p["off"], (f - np.floor(f))[stay])
