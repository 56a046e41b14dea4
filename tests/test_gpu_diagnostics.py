"""pic_moments from one packet of a launch per call: the potential's two-level scan at the
sizes around its chunks of 256 nodes and the one-block field phase's 1,024, packets too large for the pinned copy, calls that
skip arrays, and the kinetic energy over ragged particle counts."""
import ctypes as C

import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("smooth", [0, 1])
@pytest.mark.parametrize("ncells", [1, 2, 255, 256, 257, 511, 1022, 1023, 1024, 40001])
def test_diagnostics_match_the_oracle(ncells, smooth):
    """Potential and densities of the load's deposit (the oracle's field phase is exact to its
    final rounding) and the kinetic energy summed in numpy's longdouble."""
    from oracle.oracle import Oracle
    ensure_built()
    phys = W.bounded_small(ncells=ncells, ppc=3, seed=21)
    phys.smooth = smooth
    loads = W.initial_load(phys, seed=21)
    for precision, tol in ((capi.FP64, 1e-12), (capi.FP32, 2e-6)):
        sim = capi.Sim(phys, precision=precision, sort_interval=5)
        sim.load_all(loads)
        m = sim.moments(0)
        o = Oracle(phys)
        o.load_all(loads)
        om = o.moments()
        for k in ("density", "phi", "E"):
            scale = max(np.abs(om[k]).max(), 1e-300)
            np.testing.assert_allclose(m[k], om[k], rtol=0, atol=tol * scale * max(1, ncells ** 0.5))
        for s, ld in enumerate(loads):
            sp = phys.species[s]
            v2 = sum(np.asarray(v, np.longdouble) ** 2 for v in (ld.vx, ld.vy, ld.vz)).sum()
            want = float(0.5 * sp.mass * sp.weight * v2)
            # FP32: three roundings a term and that of the state, all relative and independent
            np.testing.assert_allclose(m["kinetic"][s], want, rtol=1e-13 if precision else 1e-6)
        # a call without arrays, and one with the field alone
        head = capi.pic_moments_out()
        assert capi.lib().pic_moments(sim._h, 0, C.byref(head), None, None, None) == 0
        assert list(head.live[:2]) == [3 * ncells, 3 * ncells]
        E = np.zeros(ncells + 1)
        assert capi.lib().pic_moments(sim._h, 0, C.byref(head), None, None, E.ctypes.data) == 0
        np.testing.assert_array_equal(E, m["E"])
        sim.close()
