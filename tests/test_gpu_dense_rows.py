"""Dense ingest of rows at every alignment against the oracle: widths around the 16-byte loads and the brick, a
grid that starts at an odd byte of its buffer between bytes that are not part of it, rows spread over warps by
plane (small grids) and whole (larger ones)."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(5, 3, 1), (9, 8, 15), (8, 10, 17), (17, 9, 100), (3, 20, 130), (260, 264, 33)])
@pytest.mark.parametrize("offset", [0, 1, 6])
def test_rows(shape, offset):
    import torch
    import paper_2105_04419_gb300 as V
    from paper_2105_04419_gb300.lib import _check
    rs = np.random.default_rng(sum(shape))
    occ = (rs.random(shape) < 0.01).astype(np.uint8) * rs.integers(1, 256, shape).astype(np.uint8)
    occ.flat[occ.size // 2] = 200
    buf = torch.full((occ.size + 16,), 255, dtype=torch.uint8, device="cuda")
    buf[offset:offset + occ.size] = torch.from_numpy(occ.reshape(-1)).cuda()
    torch.cuda.synchronize()
    m = V.Map(shape[2], shape[1], shape[0], 7)
    for _ in range(2):  # again over what the first left
        _check(V.load().vdbedt_set_occupancy_dense(m.handle, buf.data_ptr() + offset, 1), "dense", m.handle)
        m.global_()
        assert np.array_equal(m.export_dense(), O.edt_factorised((occ != 0).astype(np.uint8), 7))
    m.close()


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 5, 6, 7, 8])
def test_rows_narrower_than_a_brick(nx):
    """A brick plane's rows read as one stretch, at any alignment; by plane and in whole rows, the last ones short."""
    import torch
    import paper_2105_04419_gb300 as V
    from paper_2105_04419_gb300.lib import _check
    rs = np.random.default_rng(nx)
    for shape in ((1, 1, nx), (130, 13, nx), (300, 291, nx)):
        occ = (rs.random(shape) < 0.01).astype(np.uint8) * 77
        occ[shape[0] // 2, shape[1] // 2, nx // 2] = 128
        m = V.Map(nx, shape[1], shape[0], 10)
        for offset in (0, 1, 2, 3):
            buf = torch.full((occ.size + 16,), 255, dtype=torch.uint8, device="cuda")  # not part of the grid
            buf[offset:offset + occ.size] = torch.from_numpy(occ.reshape(-1)).cuda()
            torch.cuda.synchronize()
            _check(V.load().vdbedt_set_occupancy_dense(m.handle, buf.data_ptr() + offset, 1), "dense", m.handle)
            m.global_()
            assert np.array_equal(m.export_dense(), O.edt_factorised((occ != 0).astype(np.uint8), 10)), (shape, offset)
        m.close()
