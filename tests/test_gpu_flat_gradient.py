"""The distance and its gradient where all eight corners of a cell hold the same distance: exactly zero gradient
(beyond dmax, and half-way between two walls), in cells inside a brick and across its faces."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dmax,voxel", [(7, 0.1), (13, 0.3), (11, 0.07)])
def test_gradient_of_a_flat_field_is_zero(dmax, voxel):
    import paper_2105_04419_gb300 as V
    nx, ny, nz = 96, 40, 40
    occ = np.zeros((nz, ny, nx), np.uint8)
    occ[:, :, 0] = 1
    m = V.Map(nx, ny, nz, dmax, voxel_size=voxel)
    m.set_occupancy_dense(occ)
    m.global_()
    rs = np.random.default_rng(1)
    cells = np.stack([rs.integers(dmax + 1, nx - 1, 4000), rs.integers(0, ny - 1, 4000), rs.integers(0, nz - 1, 4000)], 1)
    pts = torch.as_tensor((cells + rs.random((4000, 3)) * 0.9 + 0.05) * voxel, dtype=torch.float32, device="cuda")
    d, g = m.distance_at(pts)
    assert torch.equal(g, torch.zeros_like(g))
    assert float((d - dmax * voxel).abs().max()) <= 4e-7 * dmax * voxel


@pytest.mark.parametrize("cell", [4, 7, 12])  # inside a brick, across its face
@pytest.mark.parametrize("voxel", [0.1, 0.3, 0.07])
def test_gradient_half_way_between_two_walls_is_zero(cell, voxel):
    """The cell between walls an odd number of voxels apart: eight equal distances below dmax."""
    import paper_2105_04419_gb300 as V
    nx, ny, nz = 2 * cell + 2, 40, 40
    occ = np.zeros((nz, ny, nx), np.uint8)
    occ[:, :, 0] = occ[:, :, nx - 1] = 1
    m = V.Map(nx, ny, nz, 16, voxel_size=voxel)
    m.set_occupancy_dense(occ)
    m.global_()
    rs = np.random.default_rng(cell)
    cells = np.stack([np.full(4000, cell), rs.integers(0, ny - 1, 4000), rs.integers(0, nz - 1, 4000)], 1)
    pts = torch.as_tensor((cells + rs.random((4000, 3)) * 0.9 + 0.05) * voxel, dtype=torch.float32, device="cuda")
    d, g = m.distance_at(pts)
    assert torch.equal(g, torch.zeros_like(g))
    assert float((d - cell * voxel).abs().max()) <= 4e-7 * cell * voxel
