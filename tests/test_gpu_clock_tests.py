"""Steps on which a species' clocks all test (its own steps that are multiples of 127) in the
mover's variants that draw in place: the clocks against the oracle where such a step also
sorts the store (a sort interval that divides 128), and what such a step costs."""
import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import assert_same_clocks, by_id, ensure_built, requires_gpu, run_gpu, run_oracle

pytestmark = [pytest.mark.gpu, requires_gpu]

PLASMAS = {"staged": lambda: W.bounded_small(ncells=40, ppc=70, seed=3, nu=0.2),
           "spread": lambda: W.bounded_small(ncells=300, ppc=1, seed=4, nu=0.2),
           "across segments": lambda: W.bounded_small(ncells=9, ppc=7, seed=5, nu=0.2),
           "subcycled": lambda: W.bounded_small(ncells=30, ppc=50, seed=6, nu=0.2, ion_nstep=2)}


@pytest.fixture(autouse=True)
def in_place(monkeypatch):
    """No variant of its own for these steps, whatever the size."""
    monkeypatch.setenv("BITPIC_PAIR_MIN_SLOTS", str(10 ** 9))


@pytest.mark.parametrize("kind", PLASMAS)
def test_tests_on_a_sort_step_match_the_oracle(kind):
    phys = PLASMAS[kind]()
    loads = W.initial_load(phys, seed=3)
    g, gm = run_gpu(phys, loads, 260, capi.FP64, sort_interval=8)
    o, om = run_oracle(phys, loads, 260)
    np.testing.assert_array_equal(gm["collisions"], om["collisions"])
    np.testing.assert_array_equal(gm["wall_count"], om["wall_count"])
    assert_same_clocks(g, o)


@pytest.mark.parametrize("kind", PLASMAS)
def test_tests_do_not_depend_on_the_sort(kind):
    phys = PLASMAS[kind]()
    loads = W.initial_load(phys, seed=3)
    want = [by_id(p) for p in run_gpu(phys, loads, 260, capi.FP32, sort_interval=0)[0]]
    got = [by_id(p) for p in run_gpu(phys, loads, 260, capi.FP32, sort_interval=8)[0]]
    for a, b in zip(want, got):
        for k in ("id", "cell", "off", "vx", "vy", "vz", "state"):
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
def test_cost_of_a_test_step(precision):
    """Four million particles on 256 cells.  Such a step reads an id more a particle (4 of 24 or
    40 bytes) and draws once for each: about a hundred integer instructions beside the some
    twenty of the move, so six times a plain step bounds a mover that is limited by its
    instructions throughout."""
    ensure_built()
    phys = W.bounded_small(ncells=256, ppc=8000, seed=1)
    sim = capi.Sim(phys, precision=precision, sort_interval=20, block=256)
    sim.load_all(W.initial_load(phys, seed=1))
    sim.step(121)
    sim.profile(True)
    us = []
    for _ in range(121, 132):
        before = sim.kernel_time(0)[1]
        sim.step(1)
        us.append(1e3 * (sim.kernel_time(0)[1] - before))
    sim.close()
    test = us.pop(127 - 121)
    assert test < 6.0 * np.median(us), (test, us)
