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
