"""Particles that cross more than one cell in a step: the FP64 form's common path takes them
with the others.  Positions against the oracle bit for bit around every edge of that path
(whole cells, sums that round up to 1, far beyond the cells it counts), and what a plasma of
such particles costs."""
import dataclasses

import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import (assert_same_clocks, by_id, ensure_built, particle_errors, requires_gpu,
                              run_gpu, run_oracle)

pytestmark = [pytest.mark.gpu, requires_gpu]

TINY = 2.0 ** -60
OFFSETS = [0.0, 2.0 ** -53, 0.25, 0.5, 1.0 - 2.0 ** -53]
SPEEDS = [0.0, 0.5, 1.0, 1.5, 1.75, 2.0, 3.0, 3.25, 7.5, 31.0, 4096.5, 2.0 ** 20, 2.0 ** 21 - 0.5, 2.0 ** 21,
          2.0 ** 22 + 0.25, TINY, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 2.0 + 2.0 ** -51, 3.0 + 2.0 ** -51]


def lattice(ncells):
    """Every offset with every speed of either sign, from the first, a middle and the last cell."""
    f, u, j = np.meshgrid(OFFSETS, SPEEDS + [-s for s in SPEEDS], [0, ncells // 2, ncells - 1])
    n = f.size
    z = np.zeros(n)
    return W.Load(j.ravel().astype(np.int32), f.ravel(), u.ravel(), z, z.copy(),
                  np.arange(n, dtype=np.uint32))


@pytest.mark.parametrize("sort", [0, 2])
@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_ABSORB])
@pytest.mark.parametrize("ncells", [3, 100, 9001])
def test_moves_of_any_length_match_the_oracle(ncells, bc, sort):
    load = lattice(ncells)
    phys = W.Physics(ncells=ncells, dx=1.0, dt=1.0, processes=[], bc=bc, field=W.FIELD_NONE,
                     species=[W.Species("n", 0.0, 1.0, 1.0, 0.0, 1 + len(load) // ncells, 2.0)])
    g, gm = run_gpu(phys, [load], 3, capi.FP64, sort_interval=sort)
    o, om = run_oracle(phys, [load], 3)
    np.testing.assert_array_equal(gm["wall_count"], om["wall_count"])
    a, b = by_id(g[0]), by_id(o[0])
    for k in ("id", "cell", "off"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("B", [(0.0, 0.0, 0.0), (0.3, -1.9, 0.0), (0.4, 0.5, -1.2)])
def test_a_fast_plasma_matches_the_oracle(B):
    phys = dataclasses.replace(W.bounded_small(ncells=200, ppc=40, seed=5, nu=0.05), dt=1.0, B=B,
                               bc=W.BC_PERIODIC, field=W.FIELD_NONE)
    loads = W.initial_load(phys, seed=5)
    g, gm = run_gpu(phys, loads, 30, capi.FP64, sort_interval=7)
    o, om = run_oracle(phys, loads, 30)
    np.testing.assert_array_equal(gm["collisions"], om["collisions"])
    assert_same_clocks(g, o)
    for ex, ev in particle_errors(phys, g, o):
        assert ex < 1e-12 and ev < 1e-12


def test_cost_of_fast_particles():
    """The magnetized plasma at a thermal speed of 0.8 cells a step against one of 0.1.  The FP64
    pipe bounds the push with 12 operations a particle; the floor and its subtraction make 14,
    and the deposit of tiles that have spread over more cells costs the FP32 form 17 us here,
    a fifth of this form's time: 1.17 + 0.2, and a quarter for what else may differ."""
    ensure_built()
    us = {}
    for dt in (0.05, 0.4):
        phys = dataclasses.replace(W.magnetized_source(ncells=4096, ppc=400), dt=dt)
        sim = capi.Sim(phys, precision=capi.FP64, sort_interval=20, block=256)
        sim.load_all(W.initial_load(phys, seed=1))
        sim.step(40)
        sim.profile(True)
        sim.step(20)
        n, ms = sim.kernel_time(0)
        us[dt] = 1e3 * ms / n
        sim.close()
    assert us[0.4] < 1.7 * us[0.05], us
