"""Nearest-obstacle query against the oracle's brute force in every encoding of the per-axis fields: fp16
(windowed passes), 16-bit integers (envelope passes, dmax above 45), each read back after the tuning moved to
the other form but before the next transform, and in a batch."""
import numpy as np
import pytest

import oracle as O
from gpu_common import gpu_global
from test_gpu_nearest import all_voxels

pytestmark = pytest.mark.gpu


def scattered(shape, p, seed):
    return (np.random.default_rng(seed).random(shape) < p).astype(np.uint8)


@pytest.mark.parametrize("dmax,variant,later", [(20, 0, 8), (20, 8, 3), (45, 0, 0), (46, 0, 0), (70, 0, 0)])
def test_forms(dmax, variant, later):
    occ = scattered((33, 41, 50), 0.0002, dmax)
    occ[7, 8, 9] = 1
    m = gpu_global(occ, dmax, tuning={"variant": variant} if variant else None)
    q = all_voxels(occ.shape)
    ref = O.nearest_obstacle(occ, dmax, q)
    assert np.array_equal(m.query_nearest(q), ref)
    if later:  # the stored fields keep their form until the next transform
        m.set_tuning(variant=later)
        assert np.array_equal(m.query_nearest(q), ref)
        m.global_()
        assert np.array_equal(m.query_nearest(q), ref)


def test_batch_grids():
    import paper_2105_04419_gb300 as V
    grids = [scattered(s, 0.002, i) for i, s in enumerate(((20, 33, 47), (40, 16, 24)))]
    b = V.Batch([g.shape[::-1] for g in grids], 12)
    b.set_occupancy_dense(grids)
    b.global_()
    for m, g in zip(b.maps, grids):
        q = all_voxels(g.shape)
        assert np.array_equal(m.query_nearest(q), O.nearest_obstacle(g, 12, q))


@pytest.mark.parametrize("p", [0.25, 0.45, 0.97])
@pytest.mark.parametrize("dmax", [1, 2, 8, 50])
def test_crowded_maps(p, dmax):
    """Warps whose lanes all have an obstacle within one voxel, and warps where some have not."""
    import paper_2105_04419_gb300 as V
    occ = scattered((11, 13, 19), p, dmax)
    occ[2:7, 3:8, 4:13] = 0
    m = gpu_global(occ, dmax)
    q = all_voxels(occ.shape)
    outside = q[::5] + np.array([19, 0, 0], np.int32)
    q = np.concatenate([q, outside, q[::-1]])
    assert np.array_equal(m.query_nearest(q), O.nearest_obstacle(occ, dmax, q))
    m.synchronize()
    u = V.Map(0, 0, 0, dmax, unbounded=True, max_bricks=20000, max_nodes=64)
    z, y, x = np.nonzero(occ)
    shift = np.array([-13, -10, -9], np.int32)
    u.set_occupancy(np.stack([x, y, z], 1).astype(np.int32) + shift, np.ones(len(x), np.uint8))
    u.global_()
    want = O.nearest_obstacle(occ, dmax, q[: occ.size])
    assert np.array_equal(u.query_nearest(q[: occ.size] + shift), np.where(want < 0, want, want + shift))
    u.synchronize()
