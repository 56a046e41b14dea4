"""The deposit of a species that rests on a step (subcycling, neutral particle targets)
stands from the step before.  After every step it must equal, integer by integer, the
deposit that a fresh handle forms from the same particles."""
import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


def fresh_charge(phys, sim, precision, sort):
    b = capi.Sim(phys, precision=precision, sort_interval=sort)
    for s in range(len(phys.species)):
        p = sim.particles(0, s, cell_units=True)
        b.load(0, s, W.Load(p["cell"], p["off"], p["vx"], p["vy"], p["vz"], p["id"], p["state"]),
               cell_units=True)
    raw, _ = b.charge_raw(0)
    b.close()
    return raw


def case(kind, nstep):
    if kind == "source":  # re-injection and ionization products between the moves
        return W.magnetized_source(ncells=37, ppc=21, seed=3, nu=0.4, capacity_factor=4.0,
                                   ion_nstep=nstep)
    if kind == "target":
        return W.ionization_case(ncells=33, ppc=24, nu_iz=0.2, seed=5, sort_interval=nstep)
    return W.bounded_small(ncells=29, ppc=33, seed=4, ion_nstep=nstep)


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
@pytest.mark.parametrize("kind,nstep,sort", [
    ("walls", 4, 20), ("walls", 3, 1), ("walls", 5, 7), ("source", 2, 4), ("source", 7, 5),
    ("target", 6, 6)])
def test_standing_deposit_equals_a_fresh_one(kind, nstep, sort, precision):
    ensure_built()
    phys = case(kind, nstep)
    sim = capi.Sim(phys, precision=precision, sort_interval=sort)
    sim.load_all(W.initial_load(phys, seed=7))
    for n in (1, 1, 1, 2, 1, 3, 1, 9):
        sim.step(n)
        raw, _ = sim.charge_raw(0)
        np.testing.assert_array_equal(raw, fresh_charge(phys, sim, precision, sort))
    sim.close()


def test_step_counter_set_off_the_cycle():
    """The counter set to another phase of the subcycle, without a load: the species that
    moves next is another one, and its deposit is formed anew."""
    ensure_built()
    phys = case("walls", 4)
    sim = capi.Sim(phys, precision=capi.FP64, sort_interval=20)
    sim.load_all(W.initial_load(phys, seed=7))
    sim.step(3)
    for step in (9, 6, 23):
        sim.restore_counters(step)
        for _ in range(3):
            sim.step(1)
            raw, _ = sim.charge_raw(0)
            np.testing.assert_array_equal(raw, fresh_charge(phys, sim, capi.FP64, 20))
    sim.close()
