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
