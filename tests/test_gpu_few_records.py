"""Few records on grids whose bricks mostly have storage (a flag per brick) and on grids with little storage (a sort):
the same field either way, with repeated, cleared and edge voxels, and the sort's grid refusing more bricks than fit."""
import numpy as np
import pytest

import oracle as O
from gpu_common import first_mismatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 700])
def test_flags_and_sort_agree(n):
    import paper_2105_04419_gb300 as V
    nx, ny, nz, dmax = 261, 197, 130, 10
    rs = np.random.default_rng(n)
    xyz = np.stack([rs.integers(0, 60, n), rs.integers(0, 50, n), rs.integers(0, 40, n)], 1).astype(np.int32)
    xyz[0] = (nx - 1, ny - 1, nz - 1)
    xyz[n // 2] = xyz[n - 1]
    val = (rs.random(n) < 0.9).astype(np.uint8)
    val[0] = 1
    occ = np.zeros((nz, ny, nx), np.uint8)
    for (x, y, z), v in zip(xyz, val):
        occ[z, y, x] = v
    want = O.edt_factorised(occ, dmax)
    for kw in ({}, {"max_bricks": 3500}):  # 33 x 25 x 17 = 14,025 bricks
        m = V.Map(nx, ny, nz, dmax, **kw)
        m.set_occupancy(xyz, val)
        m.global_()
        assert first_mismatch(m.export_dense(), want) is None, kw
