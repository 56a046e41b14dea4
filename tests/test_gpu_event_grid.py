"""The event kernel of a small, strongly collisional plasma: its grid follows the events of a step
and not the queue, whose size a small store bounds."""
import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
@pytest.mark.parametrize("nu", [1.0, 20.0])
def test_cost_does_not_depend_on_the_reserve(nu, precision):
    """The same events in a store of their size and in one of eight times that, whose queue is
    not bounded: the same work, and a half for the spread of such short kernels."""
    ensure_built()
    us = []
    for reserve in (1.0, 8.0):
        phys = W.bounded_small(ncells=256, ppc=127, nu=nu, seed=1)
        for s in phys.species:
            s.capacity_factor = reserve
        sim = capi.Sim(phys, precision=precision, sort_interval=20, block=256)
        sim.load_all(W.initial_load(phys, seed=1))
        sim.step(20)
        sim.profile(True)
        t = []
        for _ in range(19):
            before = sim.kernel_time(3)[1]
            sim.step(1)
            t.append(1e3 * (sim.kernel_time(3)[1] - before))
        us.append(np.median(t))
        sim.close()
    assert us[0] < 1.5 * us[1], us
