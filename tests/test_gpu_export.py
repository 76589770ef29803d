"""Dense export against the oracle's field: widths around the brick, the 16-byte store and the 128-voxel
node, ragged heights and depths, grids with unstored bricks, and an output that is only 4-byte aligned."""
import numpy as np
import pytest

import oracle as O
from gpu_common import gpu_global

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (9, 7, 4), (8, 17, 127), (17, 9, 128), (5, 24, 132), (40, 3, 257), (136, 130, 260)])
@pytest.mark.parametrize("offset", [0, 1])
def test_export_matches_oracle(shape, offset):
    import torch
    from paper_2105_04419_gb300.lib import _check, load
    rs = np.random.default_rng(sum(shape))
    occ = np.zeros(shape, np.uint8)
    at = [rs.integers(0, n, 1 + occ.size // 20000) for n in shape]
    occ[tuple(at)] = 1
    m = gpu_global(occ, 9)
    out = torch.full((occ.size + 8,), -7, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    _check(load().vdbedt_export_dense(m.handle, out.data_ptr() + 4 * offset, 1), "vdbedt_export_dense", m.handle)
    m.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got[offset:offset + occ.size].reshape(shape), O.edt_factorised(occ, 9))
    assert (got[:offset] == -7).all() and (got[offset + occ.size:] == -7).all()


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 5, 6, 7, 8])
def test_narrow_maps(nx):
    """Maps of a brick's width and less: a thread per exported voxel."""
    rs = np.random.default_rng(nx)
    for shape in ((1, 1, nx), (130, 13, nx), (9, 200, nx)):
        occ = (rs.random(shape) < 0.01).astype(np.uint8)
        m = gpu_global(occ, 10)
        assert np.array_equal(m.export_dense(), O.edt_factorised(occ, 10)), shape
        m.close()
