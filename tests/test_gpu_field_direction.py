"""The Boris push for every direction of B: in the x-y plane (the form without the z terms),
along an axis, with a z component, and beside a species without charge, against the oracle;
and a velocity that is not finite is still reported."""
import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import assert_same_clocks, ensure_built, particle_errors, requires_gpu, run_gpu, run_oracle

pytestmark = [pytest.mark.gpu, requires_gpu]

DIRECTIONS = [(2.0, 0.0, 0.0), (0.0, 1.5, 0.0), (0.3, -1.9, 0.0), (0.0, 0.0, 2.0), (0.4, 0.5, -1.2),
              (0.2, 0.0, 1e-3)]


@pytest.mark.parametrize("B", DIRECTIONS)
def test_every_direction_matches_the_oracle(B):
    phys = W.magnetized_source(ncells=64, ppc=30, seed=3, nu=0.1, capacity_factor=3.0)
    phys.B = B
    phys.species.append(W.Species("n", 0.0, 100.0, phys.species[0].weight, 0.05, 20))
    loads = W.initial_load(phys, seed=3)
    loads[0].vx[:5] = loads[0].vy[5:9] = loads[0].vz[9:12] = 0.0  # zeros of either sign on the way
    g, gm = run_gpu(phys, loads, 30, capi.FP64, sort_interval=7)
    o, om = run_oracle(phys, loads, 30)
    np.testing.assert_array_equal(gm["wall_count"], om["wall_count"])
    np.testing.assert_array_equal(gm["collisions"], om["collisions"])
    for s, (ex, ev) in enumerate(particle_errors(phys, g, o)):
        assert ex < 1e-12 and ev < 1e-12, (s, ex, ev)
    assert_same_clocks(g, o)
    g, gm = run_gpu(phys, loads, 8, capi.FP32, sort_interval=7)
    o, om = run_oracle(phys, loads, 8)
    for s, (ex, ev) in enumerate(particle_errors(phys, g, o)):
        assert ex < 1e-5 and ev < 1e-5, (s, ex, ev)


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
@pytest.mark.parametrize("B", DIRECTIONS[:4])
@pytest.mark.parametrize("component", ["vx", "vy", "vz"])
def test_a_velocity_that_is_not_finite_is_reported(component, B, precision):
    ensure_built()
    phys = W.bounded_small(ncells=16, ppc=8, seed=3)
    phys.B = B
    loads = W.initial_load(phys, seed=3)
    getattr(loads[1], component)[17] = np.inf
    sim = capi.Sim(phys, precision=precision, sort_interval=5)
    sim.load_all(loads)
    sim.step(2)
    with pytest.raises(capi.PicError) as e:
        sim.sync()
    assert e.value.code == -5
    sim.close()
