"""Whole-line passes of untruncated grids against the oracle where the staged tiles can go wrong: lines
around one brick, one group of eight bricks and the longest staged line (1,496 positions; longer ones keep
the stack kernels), x rows around one and several steps of 32 bricks, ragged across, with one far obstacle, few and many, then updates of a few voxels."""
import numpy as np
import pytest

import oracle as O
from gpu_common import coords_of, first_mismatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape_xyz", [(3, 7, 9), (9, 8, 64), (17, 63, 65), (33, 66, 8), (5, 520, 71), (6, 5, 513),
                                       (9, 1496, 3), (9, 1497, 3), (5, 3, 1495), (4, 2, 1505), (256, 5, 9),
                                       (257, 9, 2), (523, 3, 17), (2100, 2, 3)])
@pytest.mark.parametrize("count", [1, 3, 400])
def test_lines(shape_xyz, count):
    import paper_2105_04419_gb300 as V
    nx, ny, nz = shape_xyz
    rs = np.random.default_rng(nx * ny + nz + count)
    occ = np.zeros((nz, ny, nx), np.uint8)
    occ[rs.integers(0, nz, count), rs.integers(0, ny, count), rs.integers(0, nx, count)] = 1
    m = V.Map(nx, ny, nz, None)
    xyz = coords_of(occ)
    m.set_occupancy(xyz, np.ones(len(xyz), np.uint8))
    m.global_()
    for frame in range(3):
        ref = O.edt_untruncated(occ)
        got = m.export_dense()
        assert first_mismatch(got, ref) is None, (frame, first_mismatch(got, ref))
        edit = np.stack([rs.integers(0, n, 2) for n in shape_xyz], 1).astype(np.int32)
        val = np.array([1, frame & 1], np.uint8)
        for (x, y, z), v in zip(edit, val):
            occ[z, y, x] = v
        m.set_occupancy(edit, val)
        m.update()
    m.close()
