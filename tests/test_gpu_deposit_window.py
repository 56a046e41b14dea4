"""The warp's deposit of tiles that have spread over several cells, against exact integers:
charges of 0, of the whole unit (an offset that rounds up to 1) and next to it, and as many
particles of a tile in one cell as one copy of the window can see."""
import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
@pytest.mark.parametrize("span", [1, 2, 3, 4, 30, 31, 32, 33])
@pytest.mark.parametrize("offsets", ["whole", "largest", "zero", "mixed"])
def test_deposit_is_exact(offsets, span, precision):
    ensure_built()
    rng = np.random.default_rng(span)
    n, t = 5 * 128 + 77, np.float32 if precision == capi.FP32 else np.float64
    bits = 24 if precision == capi.FP32 else 48
    whole = np.nextafter(t(1), t(0)).astype(np.float64)  # FP64: its charge is the whole unit
    values = {"whole": [whole], "largest": [1.0 - 2.0 ** -bits], "zero": [0.0],
              "mixed": [whole, 1.0 - 2.0 ** -bits, 0.0, 0.5, 2.0 ** -bits, 0.3]}[offsets]
    off = rng.choice(values, n).astype(t).astype(np.float64)
    # every tile: its first and last cell once, the others crowded into one cell
    first = 3
    cell = np.full(n, first + span // 2, np.int32)
    cell[::128], cell[127::128] = first, first + span - 1
    cell[5::9] = first + rng.integers(0, span, len(cell[5::9]))
    zero = np.zeros(n)
    phys = W.Physics(ncells=40, dx=1.0, dt=1.0, processes=[], bc=W.BC_PERIODIC, field=W.FIELD_NONE,
                     species=[W.Species("n", 0.0, 1.0, 1.0, 0.0, 20, 2.0)])
    sim = capi.Sim(phys, precision=precision, sort_interval=0)
    sim.load(0, 0, W.Load(cell, off, zero, zero.copy(), zero.copy(), np.arange(n, dtype=np.uint32)))
    q = np.rint(off * 2.0 ** bits).astype(np.int64)
    want = np.zeros(41, np.int64)
    np.add.at(want, cell, (1 << bits) - q)
    np.add.at(want, cell + 1, q)
    for _ in range(2):  # the load's deposit, then a step's
        raw, unit = sim.charge_raw(0)
        assert unit == 1 << bits
        np.testing.assert_array_equal(raw[0], want)
        sim.step(1)
    sim.close()
