"""The allocation-free transform against the oracle where its passes can go wrong: rows around one and
several 640-voxel stretches (and the 192 voxels looked at beyond them), axes around eight outputs, the largest
truncation, sparse rows whose nearest obstacle lies words away."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,p,dmax", [((2, 3, 640), 0.003, 181), ((3, 2, 641), 0.002, 100), ((1, 2, 2000), 0.001, 181),
                                          ((9, 17, 33), 0.01, 7), ((7, 200, 31), 0.0005, 181), ((201, 8, 9), 0.0005, 150),
                                          ((16, 1, 1300), 0.0, 40), ((24, 25, 1), 0.02, 12)])
def test_lines(shape, p, dmax):
    import torch
    import paper_2105_04419_gb300 as V
    occ = (np.random.default_rng(sum(shape) + dmax).random(shape) < p).astype(np.uint8)
    occ[shape[0] // 2, shape[1] // 3, shape[2] // 4] = 3  # any nonzero byte is occupied
    got = V.edt_dense_noalloc(torch.from_numpy(occ).cuda(), dmax).cpu().numpy()
    assert np.array_equal(got, O.edt_factorised((occ != 0).astype(np.uint8), dmax))


@pytest.mark.parametrize("nx", [1, 2, 3, 5, 16, 17, 31, 32, 33])
@pytest.mark.parametrize("dmax", [1, 32, 33, 181])
def test_narrow_rows_and_short_lines(nx, dmax):
    """Several rows to a warp (up to 32 voxels), lines of one to nine positions along y and z."""
    import torch
    import paper_2105_04419_gb300 as V
    rs = np.random.default_rng(nx * 200 + dmax)
    for ny, nz in ((1, 1), (2, 67), (67, 2), (3, 8), (9, 3), (130, 1)):
        occ = (rs.random((nz, ny, nx)) < 0.01).astype(np.uint8)
        occ[nz // 2, ny // 3, nx // 2] = 1
        got = V.edt_dense_noalloc(torch.from_numpy(occ).cuda(), dmax).cpu().numpy()
        assert np.array_equal(got, O.edt_factorised(occ, dmax)), (ny, nz)


@pytest.mark.parametrize("shape,dmax", [((9, 1000, 200), 40), ((1, 63000, 33), 70), ((1, 2, 700), 181), ((2, 1, 129), 64),
                                        ((1, 1, 1 << 21), 65)])
def test_stretches(shape, dmax):
    """Stretches of 4 to 15 words with halos of two to six, few rows and many."""
    import torch
    import paper_2105_04419_gb300 as V
    occ = (np.random.default_rng(dmax).random(shape) < 0.002).astype(np.uint8)
    got = V.edt_dense_noalloc(torch.from_numpy(occ).cuda(), dmax).cpu().numpy()
    assert np.array_equal(got, O.edt_factorised(occ, dmax))
