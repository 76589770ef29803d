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


@pytest.mark.parametrize("max_bricks,n", [(300, 700), (300, 30), (3600, 700)])
def test_more_bricks_than_fit(max_bricks, n):
    """Sorted records whose own bricks, or whose dilation, exceed the capacity, and flagged ones (from a quarter of the
    grid's bricks on): refused at the next synchronisation, and a reset map takes what fits."""
    import paper_2105_04419_gb300 as V
    nx, ny, nz, dmax = 261, 197, 130, 10  # 14,025 bricks
    rs = np.random.default_rng(n + max_bricks)
    xyz = np.stack([rs.integers(0, k, n) for k in (nx, ny, nz)], 1).astype(np.int32)
    m = V.Map(nx, ny, nz, dmax, max_bricks=max_bricks)
    m.set_occupancy(xyz, np.ones(n, np.uint8))
    m.global_()
    with pytest.raises(V.VdbedtError) as e:
        m.synchronize()
    assert e.value.code == "EOVERFLOW"
    m.reset()
    occ = np.zeros((nz, ny, nx), np.uint8)
    occ[xyz[0, 2], xyz[0, 1], xyz[0, 0]] = 1
    m.set_occupancy(xyz[:1], np.ones(1, np.uint8))
    m.global_()
    assert first_mismatch(m.export_dense(), O.edt_factorised(occ, dmax)) is None
    m.close()
