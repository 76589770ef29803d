"""Many records at once (one flag and one mask per brick): counts around a thread's share of them, in x-row order
(runs that share a mask word), shuffled and repeated, all set or with cleared voxels among them."""
import numpy as np
import pytest

import oracle as O
from gpu_common import first_mismatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [60, 61, 63, 64, 65, 71, 255, 257, 4001])
@pytest.mark.parametrize("order", ["rows", "shuffled", "repeated", "cleared"])
def test_record_runs(n, order):
    import paper_2105_04419_gb300 as V
    nx, ny, nz, dmax = 61, 45, 37, 9
    rs = np.random.default_rng(n)
    lin = np.sort(rs.choice(nx * ny * nz, n, replace=False))
    if order == "rows":
        start = rs.integers(0, nx * ny * nz - n)
        lin = np.arange(start, start + n)
    if order == "shuffled":
        rs.shuffle(lin)
    if order == "repeated":
        lin = np.repeat(lin[: (n + 2) // 3], 3)[:n]
    val = np.ones(n, np.uint8)
    if order == "cleared":
        lin = np.concatenate([lin[: n - n // 4], rs.permutation(lin)[: n // 4]])
        val[n - n // 4:] = 0
    xyz = np.stack([lin % nx, lin // nx % ny, lin // (nx * ny)], 1).astype(np.int32)
    occ = np.zeros((nz, ny, nx), np.uint8)
    for (x, y, z), v in zip(xyz, val):
        occ[z, y, x] = v
    m = V.Map(nx, ny, nz, dmax)
    m.set_occupancy(xyz, val)
    m.global_()
    assert first_mismatch(m.export_dense(), O.edt_factorised(occ, dmax)) is None
