"""The mover's variants of large batches, forced on small ones: tiles fetched ahead, warps
taking chunks of consecutive tiles, and the variant of the steps on which every clock
tests.  Each gives the particles, clocks, counters and fields of the plain variant bit for
bit, at sizes around a tile (128 particles) and a chunk, across segments, walls, sorts and
step 127."""
import dataclasses

import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import by_id, ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

VARIANTS = {"ahead": (0, 10 ** 9, 10 ** 9), "chunks": (0, 0, 10 ** 9), "full": (10 ** 9, 10 ** 9, 0),
            "all": (0, 0, 0)}


def plasmas(kind):
    if kind == "ragged":  # one particle, around one tile, around a chunk of 8 tiles, many
        sizes = [(1, 1), (1, 127), (1, 129), (43, 3), (31, 33), (33, 32), (257, 41)]
        return [W.bounded_small(ncells=n, ppc=p, seed=11 + i) for i, (n, p) in enumerate(sizes)]
    if kind == "fast":  # a quarter of the electrons and more cross a cell edge in a step
        return [dataclasses.replace(W.bounded_small(ncells=61, ppc=67, seed=2), dt=0.4)]
    if kind == "mixed":  # magnetized beside unmagnetized, volume source and ionization
        return [W.magnetized_source(ncells=53, ppc=29, seed=3, nu=0.2, capacity_factor=3.0),
                W.bounded_small(ncells=40, ppc=50, seed=4)]
    if kind == "subcycled":
        return [W.bounded_small(ncells=61, ppc=45, seed=5, ion_nstep=4),
                W.bounded_small(ncells=17, ppc=30, seed=6)]
    return [W.ionization_case(ncells=96, ppc=48, nu_iz=0.1, seed=7, sort_interval=6)]


def result(physs, precision, sort, steps):
    sim = capi.Sim(physs, precision=precision, sort_interval=sort, block=128)
    for i, p in enumerate(physs):
        sim.load_all(W.initial_load(p, seed=p.seed), inst=i)
    for n in steps:
        sim.step(n)
    out = []
    for i, p in enumerate(physs):
        out.append(sim.charge_raw(i)[0])
        m = sim.moments(i)
        out += [m[k] for k in ("live", "wall_count", "collisions", "phi", "E")]
        for s in range(len(p.species)):
            part = by_id(sim.particles(i, s, cell_units=True))
            out += [part[k] for k in ("id", "cell", "off", "vx", "vy", "vz", "state")]
    sim.close()
    return out


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
@pytest.mark.parametrize("kind", ["ragged", "fast", "mixed", "subcycled", "target"])
def test_variants_give_the_plain_result(kind, precision, monkeypatch):
    ensure_built()
    physs = plasmas(kind)
    sort = 6 if kind == "target" else 7
    steps = (1, 30, 99) if kind != "fast" else (1, 12)
    for name in ("BITPIC_AHEAD_TILES", "BITPIC_CHUNK_ROUNDS", "BITPIC_PAIR_MIN_SLOTS"):
        monkeypatch.setenv(name, str(10 ** 9))
    want = result(physs, precision, sort, steps)
    for variant, env in VARIANTS.items():
        for name, v in zip(("BITPIC_AHEAD_TILES", "BITPIC_CHUNK_ROUNDS", "BITPIC_PAIR_MIN_SLOTS"), env):
            monkeypatch.setenv(name, str(v))
        for a, b in zip(want, result(physs, precision, sort, steps)):
            np.testing.assert_array_equal(a, b, err_msg=variant)
