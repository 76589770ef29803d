"""The envelope form's x pass on rows whose nearest obstacles lie many bricks away (up to dmax 181), with sides
that are no multiples of a brick or a run: against the oracle."""
import numpy as np
import pytest

import oracle as O
from gpu_common import first_mismatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dmax", [46, 64, 65, 100, 181])
@pytest.mark.parametrize("count", [1, 3, 40])
def test_far_obstacles_in_a_row(dmax, count):
    import paper_2105_04419_gb300 as V
    rs = np.random.default_rng(dmax + count)
    nz, ny, nx = 10, 13, 421
    occ = np.zeros((nz, ny, nx), np.uint8)
    for z, y, x in zip(rs.integers(0, nz, count), rs.integers(0, ny, count), rs.integers(0, nx, count)):
        occ[z, y, x] = 1
    m = V.Map(nx, ny, nz, dmax)
    m.set_occupancy_dense(occ)
    m.global_()
    got = m.export_dense()
    assert first_mismatch(got, O.edt_factorised(occ, dmax)) is None
