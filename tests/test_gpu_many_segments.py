"""Batches of very many small instances: the tile list that the field phase builds for the next
step, over more segments than a block has threads, and what it costs."""
import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import by_id, ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def state(sim, i):
    m = sim.moments(i)
    out = [m[k] for k in ("live", "wall_count", "collisions", "phi", "E")]
    for s in range(2):
        p = by_id(sim.particles(i, s, cell_units=True))
        out += [p[k] for k in ("id", "cell", "off", "vx", "state")]
    return out


@pytest.mark.parametrize("cells,ninst", [(3, 127), (3, 129), (3, 1025), (40, 700), (1030, 300)])
def test_every_instance_matches_its_own_run(cells, ninst):
    """Uneven segments, some of them empty: each instance as if alone, bit for bit."""
    ensure_built()
    physs = [W.bounded_small(ncells=cells, ppc=1 + 7 * i % 5, seed=1 + i) for i in range(ninst)]
    loads = [W.initial_load(p, seed=1 + i) for i, p in enumerate(physs)]
    batch = capi.Sim(physs, precision=capi.FP64, sort_interval=7)
    for i, ld in enumerate(loads):
        if i % 6:
            batch.load_all(ld, inst=i)
    batch.step(30)
    for i in sorted({0, 1, 6, 31, 64, ninst // 2, ninst - 2, ninst - 1}):
        one = capi.Sim(physs[i], precision=capi.FP64, sort_interval=7)
        if i % 6:
            one.load_all(loads[i])
        one.step(30)
        for a, b in zip(state(batch, i), state(one, 0)):
            np.testing.assert_array_equal(a, b, err_msg=str(i))
        one.close()
    batch.close()


def test_cost_of_the_tile_list():
    """The field phase of 1,000 instances of 31 cells beside that of one.  Its blocks run side by
    side; the list of 2,000 segments adds, in one block, a dozen dependent accesses to
    memory at a microsecond or so and its scan: 20 us bound it."""
    ensure_built()
    us = []
    for ninst in (1, 1000):
        physs = [W.bounded_small(ncells=31, ppc=50, seed=1 + i) for i in range(ninst)]
        sim = capi.Sim(physs, precision=capi.FP32, sort_interval=20, block=256)
        loads = W.initial_load(physs[0], seed=1)
        for i in range(ninst):
            sim.load_all(loads, inst=i)
        sim.step(40)
        sim.profile(True)
        sim.step(20)
        n, ms = sim.kernel_time(1)
        us.append(1e3 * ms / n)
        sim.close()
    assert us[1] < us[0] + 20.0, us
