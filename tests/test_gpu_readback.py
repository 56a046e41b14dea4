"""Reading particles back to host memory: pinned outputs large enough for several chunks of
write and copy, pageable ones whole, mixed and fresh memory, every array against the others;
and what memory that was never touched costs."""
import ctypes as C
import mmap
import time

import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

NAMES = ("cell", "off", "vx", "vy", "vz", "id", "state")


def types(dtype):
    return (np.int32, dtype, dtype, dtype, dtype, np.uint32, np.uint8)


def pinned(n, dtype):
    import torch
    return torch.empty(n * np.dtype(dtype).itemsize, dtype=torch.uint8, pin_memory=True).numpy().view(dtype)


def fresh(n, dtype):
    """An array of its own anonymous mapping, none of its pages touched."""
    size = n * np.dtype(dtype).itemsize
    return np.frombuffer(mmap.mmap(-1, size), np.uint8)[:size].view(dtype)


def read(sim, n, arrays, dtype):
    fn = capi.lib().pic_get_particles_f32 if dtype == np.float32 else capi.lib().pic_get_particles
    got = C.c_int64()
    t = time.perf_counter()
    rc = fn(sim._h, 0, 0, n, *[None if a is None else a.ctypes.data for a in arrays], capi.CELL_UNITS,
            C.byref(got))
    t = time.perf_counter() - t
    assert rc == 0 and got.value == n
    return t


def plasma(cells, ppc, precision):
    """Electrons with holes in their segment (walls) and a ragged last block of slots."""
    ensure_built()
    phys = W.bounded_small(ncells=cells, ppc=ppc, seed=3)
    sim = capi.Sim(phys, precision=precision, sort_interval=20)
    sim.load_all(W.initial_load(phys, seed=3))
    sim.step(7)
    return sim, sim.count(0, 0)


@pytest.mark.parametrize("precision", [capi.FP32, capi.FP64])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("cells,ppc", [(61, 17), (2003, 199)])
def test_every_kind_of_memory_gets_the_same(cells, ppc, dtype, precision):
    sim, n = plasma(cells, ppc, precision)
    want = [np.zeros(n, t) for t in types(dtype)]
    read(sim, n, want, dtype)
    assert len(np.unique(want[5])) == n  # every particle once
    some = (0, 2, 5)
    for kinds in ([pinned] * 7, [fresh] * 7, [pinned if k % 2 else fresh for k in range(7)],
                  [pinned if k in some else None for k in range(7)]):
        out = [None if f is None else f(n, t) for f, t in zip(kinds, types(dtype))]
        for a in out:
            if a is not None and kinds[0] is not fresh:
                a.view(np.uint8)[:] = 0xA5
        read(sim, n, out, dtype)
        for name, a, b in zip(NAMES, out, want):
            if a is not None:
                np.testing.assert_array_equal(a.view(np.uint8), b.view(np.uint8), err_msg=name)
    # unaligned to pages, and nothing past the end written
    pad = [np.full(n + 64, 7, t) for t in types(dtype)]
    read(sim, n, [a[32:32 + n] for a in pad], dtype)
    for a, b in zip(pad, want):
        np.testing.assert_array_equal(a[32:32 + n].view(np.uint8), b.view(np.uint8))
        assert (a[:32] == 7).all() and (a[32 + n:] == 7).all()
    sim.close()


def test_cost_of_fresh_memory():
    """Two million particles, 82 MB of double-precision outputs, into new arrays, most of whose
    memory was never touched.  The kernel clears it at ten gigabytes a second or more (0.1 ms
    a MB) and the link copies it at a hundred; 0.15 ms a MB bounds both with what else the
    call does."""
    sim, n = plasma(10000, 200, capi.FP64)
    size = sum(np.dtype(t).itemsize for t in types(np.float64)) * n / 2 ** 20
    ms, kept = [], []  # (kept: the allocator would hand out the same memory again)
    for _ in range(5):
        kept.append([np.zeros(n, t) for t in types(np.float64)])
        ms.append(1e3 * read(sim, n, kept[-1], np.float64))
    sim.close()
    assert np.median(ms) < 0.15 * size, (ms, size)
