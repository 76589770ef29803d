"""The runs that an incremental update recomputes, against a brute-force count on the CPU.

On a map whose bricks are all stored, the dirty runs of an update are those holding a brick within the
truncation distance of a changed brick: in space (z runs), in its brick layer (y runs), in its brick row
(x runs).  Run lengths 4, 8 and 16, radii from one brick to the windowed form's largest, sides that end
inside a brick, a run and a node, edits in the corners; one changed brick, some, and more than the
launch has blocks for (a thread per row instead of a block per changed brick).  The field after each
update is the fresh transform's.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def gap2(a, b):
    d = np.abs(a - b)
    return np.where(d == 0, 0, 8 * d - 7) ** 2


def expected_runs(changed, dims, dmax, runs):
    """Dirty runs per axis of changed bricks (x, y, z) on a map of dims bricks, all stored."""
    bx, by, bz = (np.arange(n) for n in dims)
    dirty = [np.zeros([dims[2], dims[1], dims[0]], bool) for _ in range(3)]
    for cx, cy, cz in changed:
        gx, gy, gz = gap2(bx, cx), gap2(by, cy), gap2(bz, cz)
        dirty[2] |= gz[:, None, None] + gy[None, :, None] + gx[None, None, :] < dmax * dmax
        dirty[1][cz] |= gy[:, None] + gx[None, :] < dmax * dmax
        dirty[0][cz, cy] |= gx < dmax * dmax
    out = []
    for axis, run in enumerate(runs):
        d = np.moveaxis(dirty[axis], 2 - axis, -1)
        pad = -d.shape[-1] % run
        d = np.pad(d, [(0, 0), (0, 0), (0, pad)])
        out.append(int(d.reshape(d.shape[0], d.shape[1], -1, run).any(-1).sum()))
    return out


def filled_map(shape, dmax, seed, runs):
    import paper_2105_04419_gb300 as V
    nz, ny, nx = shape
    g = torch.Generator(device="cuda").manual_seed(seed)
    occ = (torch.rand(shape, device="cuda", generator=g) < 0.02).to(torch.uint8)
    occ[3::8, 3::8, 3::8] = 1  # an obstacle in every whole brick
    m = V.Map(nx, ny, nz, dmax)
    m.set_tuning(x_run=runs[0], y_run=runs[1], z_run=runs[2])
    m.set_occupancy_dense(occ)
    m.global_()
    return m, occ


def check(m, occ, xyz, dmax, runs):
    import paper_2105_04419_gb300 as V
    nz, ny, nx = occ.shape
    x = torch.as_tensor(xyz, device="cuda", dtype=torch.int32)
    now = occ[x[:, 2].long(), x[:, 1].long(), x[:, 0].long()]
    m.set_occupancy(x, 1 - now)
    st = m.update(stats=True)
    occ[x[:, 2].long(), x[:, 1].long(), x[:, 0].long()] = 1 - now
    dims = [-(-n // 8) for n in (nx, ny, nz)]
    want = expected_runs(np.unique(xyz >> 3, axis=0), dims, dmax, runs)
    if not st["global_form"]:
        assert [st["x_items"], st["y_items"], st["z_items"]] == want
    f = V.Map(nx, ny, nz, dmax)
    f.set_occupancy_dense(occ)
    f.global_()
    assert torch.equal(m.export_dense(on_device=True), f.export_dense(on_device=True))
    return st


@pytest.mark.parametrize("dmax", [3, 8, 9, 32, 45])
@pytest.mark.parametrize("runs", [(4, 4, 4), (8, 16, 4), (16, 4, 8)])
def test_dirty_runs(dmax, runs):
    shape = (141, 203, 262)
    m, occ = filled_map(shape, dmax, dmax, runs)
    nz, ny, nx = shape
    rs = np.random.default_rng(dmax)
    check(m, occ, np.array([[131, 100, 70]]), dmax, runs)  # one brick beside a node's edge
    corners = np.array([[x, y, z] for x in (0, nx - 1) for y in (0, ny - 1) for z in (0, nz - 1)])
    check(m, occ, corners, dmax, runs)
    some = np.unique(np.stack([rs.integers(0, n, 25) for n in (nx, ny, nz)], 1), axis=0)
    check(m, occ, some, dmax, runs)
    st = check(m, occ, some[:1], dmax, runs)  # nothing left over from the updates before
    assert not st["global_form"]


def test_dirty_runs_of_many_bricks():
    """More changed bricks than twice the launch's blocks, in the incremental form."""
    shape, dmax, runs = (400, 512, 512), 8, (4, 8, 4)
    m, occ = filled_map(shape, dmax, 5, runs)
    bricks = np.stack(np.meshgrid(np.arange(40), np.arange(40), np.arange(4, 8)), -1).reshape(-1, 3)  # 6400 bricks
    st = check(m, occ, bricks * 8 + 2, dmax, runs)
    assert st["changed_bricks"] == 6400 and not st["global_form"]
    st = check(m, occ, bricks[:3] * 8 + 5, dmax, runs)
    assert st["changed_bricks"] == 3


def test_dirty_runs_of_a_batch():
    import paper_2105_04419_gb300 as V
    dmax, runs, shapes = 24, (4, 4, 4), [(70, 90, 131), (40, 130, 66), (129, 33, 100)]
    g = torch.Generator(device="cuda").manual_seed(1)
    occ = []
    for s in shapes:
        o = (torch.rand(s, device="cuda", generator=g) < 0.02).to(torch.uint8)
        o[3::8, 3::8, 3::8] = 1
        occ.append(o)
    b = V.Batch([s[::-1] for s in shapes], dmax)
    b.set_occupancy_dense(occ)
    b.global_()
    rs = np.random.default_rng(2)
    for n in (1, 2, 1):
        want = np.zeros(3, int)
        for i, (nz, ny, nx) in enumerate(shapes):
            xyz = np.unique(np.stack([rs.integers(0, k, n) for k in (nx, ny, nz)], 1), axis=0)
            x = torch.as_tensor(xyz, device="cuda", dtype=torch.int32)
            at = (x[:, 2].long(), x[:, 1].long(), x[:, 0].long())
            b.maps[i].set_occupancy(x, 1 - occ[i][at])
            occ[i][at] = 1 - occ[i][at]
            want += expected_runs(np.unique(xyz >> 3, axis=0), [-(-k // 8) for k in (nx, ny, nz)], dmax, runs)
        st = b.update(stats=True)
        if not any(s["global_form"] for s in st):
            assert [st[0]["x_items"], st[0]["y_items"], st[0]["z_items"]] == list(want)
        for i, (nz, ny, nx) in enumerate(shapes):
            f = V.Map(nx, ny, nz, dmax)
            f.set_occupancy_dense(occ[i])
            f.global_()
            assert torch.equal(b.maps[i].export_dense(on_device=True), f.export_dense(on_device=True))


@pytest.mark.parametrize("dmax", [17, 24, 32, 45])
def test_whole_transform_runs(dmax):
    """A map large enough for the longer runs, ragged on every axis, against runs of 4 and of 16."""
    import paper_2105_04419_gb300 as V
    nz, ny, nx = 205, 333, 421
    g = torch.Generator(device="cuda").manual_seed(dmax)
    occ = (torch.rand((nz, ny, nx), device="cuda", generator=g) < 1e-5).to(torch.uint8)
    fields = []
    for run in (0, 4, 16):
        m = V.Map(nx, ny, nz, dmax)
        m.set_tuning(x_run=run, y_run=run, z_run=run)
        m.set_occupancy_dense(occ)
        m.global_()
        fields.append(m.export_dense(on_device=True))
    assert torch.equal(fields[0], fields[1]) and torch.equal(fields[0], fields[2])
