"""The diagnostics' device packet is sized by the instances of the batch."""
import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from paper_2404_10270_gb300 import workloads as W
from tests.gpu_common import ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]

NODES = 4_000_001


def memory(field, nspecies, bc):
    import torch
    phys = W.Physics(ncells=NODES - 1, dx=0.5, dt=0.05, processes=[], field=field, bc=bc,
                     species=[W.Species("n%d" % k, (-1.0) ** k, 1.0, 1.0, 1.0, 0) for k in range(nspecies)])
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sim = capi.Sim(phys, precision=capi.FP32, sort_interval=20, block=256, capacity=[[64] * nspecies])
    used = free - torch.cuda.mem_get_info()[0]
    m = sim.moments(0)
    assert m["density"].shape == (nspecies, NODES) and not m["density"].any()
    assert m["E"].shape == (NODES,) and m["phi"].shape == (NODES,)
    sim.close()
    return used


def test_packet_follows_the_species():
    """Per node and species: accelerations 8 bytes, two deposits 16, the histogram 4; E 8 per
    node; the field's chunk sums under one.  The packet may add a density per species, E and
    (with a field solve) the potential, and an allocation's granule of 2 MB each for some
    forty arrays."""
    ensure_built()
    for field, bc, nspecies, values in ((W.FIELD_NONE, W.BC_PERIODIC, 1, 2), (W.FIELD_POISSON, W.BC_ABSORB, 1, 3),
                                        (W.FIELD_POISSON, W.BC_ABSORB, 4, 6)):
        bound = NODES * (28 * nspecies + 8 + 1 + 8 * values) + (80 << 20)
        used = memory(field, nspecies, bc)
        assert used < bound, (field, nspecies, used / NODES, bound / NODES)
