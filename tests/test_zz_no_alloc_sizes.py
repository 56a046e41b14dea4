"""pic_field_solve_noalloc at the sizes around its one-block solve and its chunks of 256
nodes, against the same formula in exact Python integers (one rounding to double)."""
import ctypes as C

import numpy as np
import pytest

from paper_2404_10270_gb300 import capi
from tests.gpu_common import ensure_built, requires_gpu

pytestmark = [pytest.mark.gpu, requires_gpu]


@pytest.mark.parametrize("ncells", [1, 2, 30, 31, 32, 254, 255, 1022, 1023, 1024, 1279, 1280, 4097,
                                    65535, 65536])
@pytest.mark.parametrize("unit", [1 << 24, 1 << 48])
def test_field_is_the_exact_one(ncells, unit):
    import torch
    ensure_built()
    rng = np.random.default_rng(ncells)
    charge = rng.integers(0, 3000 * unit, size=(3, ncells + 1), dtype=np.int64)
    z = [-1, 1, 3]
    d = torch.from_numpy(charge.reshape(-1)).cuda()
    E = torch.full((ncells + 1,), float("nan"), dtype=torch.float64, device="cuda")
    rc = capi.lib().pic_field_solve_noalloc(ncells, 3, d.data_ptr(), (C.c_int32 * 3)(*z), 0.25, unit,
                                            0.5, E.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0, capi.lib().pic_last_error(None)
    torch.cuda.synchronize()
    n = ncells
    Z = [sum(z[k] * int(charge[k, j]) for k in range(3)) for j in range(n + 1)]
    U = sum((n - j) * Z[j] for j in range(1, n))
    lam = 0.25 / (2.0 * float(n) * float(unit) * 0.5)
    want, R = np.empty(n + 1), 0  # R: sum of Z over the interior nodes before j
    for j in range(n + 1):
        if j == 0:
            G = -2 * U - 2 * n * Z[0]
        elif j == n:
            G = 2 * n * R - 2 * U + 2 * n * Z[n]
        else:
            G = n * (2 * R + Z[j]) - 2 * U
            R += Z[j]
        want[j] = lam * float(G)
    np.testing.assert_array_equal(E.cpu().numpy(), want)
