"""The mover's walks over the tiles of a batch, with its grid held to a few blocks so that each
warp takes many tiles: the resident grid's stride, fixed chunks and the chunks of batches of
short segments, direct and fetched ahead, across segments, empty and resting ones, and on
the steps that count, sort and test.  Each gives the plain result (a tile a warp) bit for
bit; and what a batch of many instances costs beside one instance of its size."""
import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import ensure_built, requires_gpu
from tests.test_gpu_mover_variants import plasmas, result

pytestmark = [pytest.mark.gpu, requires_gpu]

OFF = 10 ** 9


def batch(kind):
    if kind == "long":  # two segments of 60 tiles each
        return [W.bounded_small(ncells=120, ppc=64, seed=12)]
    if kind == "short":  # segments of one to eight tiles, resting ions in every other instance
        return [W.bounded_small(ncells=20 + 7 * i, ppc=6 + 9 * i % 23, seed=20 + i,
                                ion_nstep=1 + 3 * (i % 2)) for i in range(9)]
    return plasmas(kind)


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
@pytest.mark.parametrize("kind", ["long", "short", "ragged", "mixed", "subcycled", "target"])
def test_walks_give_the_plain_result(kind, precision, monkeypatch):
    ensure_built()
    physs = batch(kind)
    sort = 6 if kind == "target" else 7
    steps = (1, 30, 99)

    def run(blocks, ahead, chunks, full):
        for name, v in (("MOVE_BLOCKS", blocks), ("AHEAD_TILES", ahead), ("CHUNK_ROUNDS", chunks),
                        ("PAIR_MIN_SLOTS", full)):
            monkeypatch.setenv("BITPIC_" + name, str(v))
        return result(physs, precision, sort, steps)

    want = run(0, OFF, OFF, OFF)
    for blocks in (1, 3):
        for ahead in (0, OFF):
            for chunks in (0, OFF):
                for full in (0, OFF):
                    for a, b in zip(want, run(blocks, ahead, chunks, full)):
                        np.testing.assert_array_equal(a, b, err_msg=str((blocks, ahead, chunks, full)))


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
def test_cost_of_many_instances(precision):
    """500 instances of 100 cells against one of 50,000, 20 M particles either way: the same
    bytes and operations.  A warp enters a segment every eight tiles or so instead of
    never; waiting for its constants is a fifth of a tile's time at most, so 1.3 bounds it."""
    ensure_built()
    us = []
    for ni, cells in ((1, 50000), (500, 100)):
        physs = [W.bounded_small(ncells=cells, ppc=200, seed=1 + i) for i in range(ni)]
        sim = capi.Sim(physs, precision=precision, sort_interval=20, block=256)
        loads = W.initial_load(physs[0], seed=1)
        for i in range(ni):
            sim.load_all(loads, inst=i)
        sim.step(40)
        sim.profile(True)
        sim.step(20)
        n, ms = sim.kernel_time(0)
        us.append(1e3 * ms / n)
        sim.close()
    assert us[1] < 1.3 * us[0], us
