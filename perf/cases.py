"""The work that is timed: what users of the library have it do, through its public entry points.

Listed cases, and what each stands for:

  cube_64            a small dense map transformed and read whole (the 64^3 parity cube, dmax 16): the
                     smallest calls, where launches and latency count
  noalloc_ragged     the allocation-free call on a small ragged dense grid, as a control loop makes it
  tunnel_1024        the headline scene (1024 x 1024 x 256, dmax 32): reset, occupancy records from
                     device memory, global transform, the whole field
  tunnel_host_masks  the end-to-end form: occupied bricks as bit masks from page-locked host memory,
                     transform, distances of 2^20 voxels back to host memory
  tunnel_dmax64      a larger truncation than the windowed passes serve (lower-envelope passes)
  tunnel_untruncated the paper's dmax = infinity on a whole map
  lidar_session      online mapping: a map built from lidar frames, an update and a local query each
  lidar_untruncated  the same without truncation
  edits_ablation     the paper's ablation: a share of the obstacles moved and moved back, as a
                     captured update
  batch_16           maps of uneven size (dmax 24) transformed together, then edited together
  planner_points     trajectories: clearance cost and its gradient, distances and gradients at points
  nearest_voxels     nearest obstacle of voxels all over a map

Scenes are seeded and made on the GPU: spline tunnels (walls of 1.5 voxels around tubes of radius 8 to
24), lidar frames cast in them, uneven random cubes with boxes.
"""
import math

import numpy as np
import torch

import paper_2105_04419_gb300 as V

DEV = "cuda"


def listed():
    return [
        dict(name="cube_64", kind="dense", nx=64, ny=64, nz=64, dmax=16, p=0.02),
        dict(name="noalloc_ragged", kind="noalloc", nx=117, ny=96, nz=83, dmax=24, p=0.004),
        dict(name="tunnel_1024", kind="tunnel", nx=1024, ny=1024, nz=256, dmax=32, tunnels=40),
        dict(name="tunnel_host_masks", kind="host_masks", nx=512, ny=512, nz=256, dmax=32, tunnels=16, queries=1 << 20),
        dict(name="tunnel_dmax64", kind="tunnel", nx=512, ny=512, nz=256, dmax=64, tunnels=16),
        dict(name="tunnel_untruncated", kind="tunnel", nx=512, ny=512, nz=256, dmax=0, tunnels=16),
        dict(name="lidar_session", kind="lidar", nx=1024, ny=1024, nz=256, dmax=32, tunnels=40, frames=12),
        dict(name="lidar_untruncated", kind="lidar", nx=512, ny=512, nz=256, dmax=0, tunnels=16, frames=6),
        dict(name="edits_ablation", kind="edits", nx=512, ny=512, nz=256, dmax=32, tunnels=16, share=0.001),
        dict(name="batch_16", kind="batch", maps=16, smin=32, smax=512, step=8, dmax=24, records=2000),
        dict(name="planner_points", kind="points", nx=512, ny=512, nz=256, dmax=32, tunnels=16, traj=8192, pts=128),
        dict(name="nearest_voxels", kind="nearest", nx=512, ny=512, nz=256, dmax=32, tunnels=16, queries=1 << 20),
    ]


def draw(rng):
    """One more case of the listed ones' kinds; sizes over the whole range, mostly not multiples of 8."""
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    kind = rng.choice(["dense", "noalloc", "tunnel", "tunnel", "tunnel", "host_masks", "lidar", "edits", "batch",
                       "points", "nearest"])
    if kind == "dense":
        return dict(kind=kind, nx=log(40, 300), ny=log(40, 300), nz=log(24, 200), dmax=rng.randint(4, 45),
                    p=round(math.exp(rng.uniform(math.log(0.001), math.log(0.05))), 5))
    if kind == "noalloc":
        return dict(kind=kind, nx=log(20, 128), ny=log(20, 128), nz=log(20, 128), dmax=rng.randint(4, 60),
                    p=round(math.exp(rng.uniform(math.log(0.001), math.log(0.05))), 5))
    if kind == "batch":
        return dict(kind=kind, maps=rng.randint(3, 20), smin=24, smax=log(64, 400), step=rng.choice([1, 8]),
                    dmax=rng.randint(6, 40), records=log(50, 4000))
    c = dict(kind=kind, nx=log(150, 900), ny=log(150, 900), nz=log(90, 256))
    c["tunnels"] = max(4, c["nx"] * c["ny"] * c["nz"] // 6_000_000)
    c["dmax"] = rng.randint(8, 45)
    if kind == "tunnel":
        form = rng.choice(["windowed", "large", "none"])
        c["dmax"] = dict(windowed=c["dmax"], large=rng.randint(46, 181), none=0)[form]
    elif kind == "host_masks":
        c["queries"] = log(1 << 12, 1 << 20)
    elif kind == "lidar":
        c["dmax"] = rng.choice([c["dmax"], 0])
        c["frames"] = rng.randint(3, 10 if c["dmax"] else 5)
    elif kind == "edits":
        c["share"] = round(math.exp(rng.uniform(math.log(1e-4), math.log(0.1))), 6)
    elif kind == "points":
        c["traj"], c["pts"] = log(64, 8192), log(16, 200)
    else:
        c["queries"] = log(1 << 12, 1 << 20)
    return c


# ---- scenes (made on the GPU from the seed) ----
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _tunnel_scene(case, seed):
    """Wall occupancy [nz, ny, nx] uint8 (a voxel is wall when the nearest tube's surface lies 0 to 1.5
    voxels further in) and the first tunnel's centre line."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    r = np.random.default_rng([int(seed), 1])
    dims = np.array([nx, ny, nz], dtype=np.float64)
    depth = torch.full((nz, ny, nx), 1e6, dtype=torch.float32, device=DEV)
    first = None
    for k in range(case["tunnels"]):
        rad = r.uniform(8, 24)
        rad = min(rad, 0.2 * dims.min())
        lo, hi = np.full(3, rad + 2), dims - rad - 3
        ctl = lo + (hi - lo) * r.random((5, 3))
        p = np.concatenate([2 * ctl[:1] - ctl[1:2], ctl, 2 * ctl[-1:] - ctl[-2:-1]])
        t = (np.arange(16) / 16.0)[:, None]
        line = [0.5 * (2 * p[i + 1] + t * (p[i + 2] - p[i]) + t * t * (2 * p[i] - 5 * p[i + 1] + 4 * p[i + 2] - p[i + 3])
                       + t ** 3 * (3 * p[i + 1] - p[i] - 3 * p[i + 2] + p[i + 3])) for i in range(4)]
        line = np.clip(np.concatenate(line + [ctl[-1:]]), lo, hi)
        first = line if first is None else first
        for a, b in zip(line[:-1], line[1:]):
            l0 = np.maximum(np.floor(np.minimum(a, b) - rad - 2), 0).astype(int)
            h0 = np.minimum(np.ceil(np.maximum(a, b) + rad + 3), dims).astype(int)
            d, dd = b - a, max(float(((b - a) ** 2).sum()), 1e-9)
            x, y, z = (torch.arange(l0[i], h0[i], device=DEV, dtype=torch.float32) - float(a[i]) for i in range(3))
            x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
            u = ((x * float(d[0]) + y * float(d[1]) + z * float(d[2])) / dd).clamp_(0, 1)
            dist = ((x - u * float(d[0])).square() + (y - u * float(d[1])).square()
                    + (z - u * float(d[2])).square()).sqrt_().sub_(rad)
            box = depth[l0[2]:h0[2], l0[1]:h0[1], l0[0]:h0[0]]
            torch.minimum(box, dist, out=box)
    occ = ((depth >= 0) & (depth < 1.5)).to(torch.uint8)
    return occ, first


def _random_map(side, seed, p, boxes):
    g = _gen(seed)
    occ = (torch.rand((side, side, side), device=DEV, generator=g) < p).to(torch.uint8)
    r = np.random.default_rng([int(seed), 2])
    for _ in range(boxes):
        size = r.integers(2, max(3, side // 4), 3)
        at = [int(r.integers(0, side - s + 1)) for s in size]
        occ[at[0]:at[0] + size[0], at[1]:at[1] + size[1], at[2]:at[2] + size[2]] = 1
    return occ


def _coords(occ):
    """[n, 3] int32 (x, y, z) of the occupied voxels, in linear order."""
    return occ.nonzero().flip(1).to(torch.int32).contiguous()


def _split(lin, nx, ny):
    return torch.stack([lin % nx, lin // nx % ny, lin // (nx * ny)], -1).to(torch.int32)


def _voxels(case, n, seed):
    g = _gen(seed)
    return torch.stack([torch.randint(0, case[k], (n,), device=DEV, generator=g, dtype=torch.int32)
                        for k in ("nx", "ny", "nz")], 1)


def _lidar_frames(case, seed, truth, line):
    """Edit records of `frames` scans along the centre line: 64 x 1024 rays walked to the first wall voxel
    (at most 400 voxels).  A ray clears the voxels it passes that the map holds occupied, then sets its
    hit; 1 in 100 hits is missed and 1 in 100 rays sets a voxel it passes."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    g = _gen(seed + 77)
    held = torch.zeros(truth.numel(), dtype=torch.uint8, device=DEV)
    seen = truth.view(-1)
    el = torch.linspace(-22.5, 22.5, 64, device=DEV).deg2rad()[:, None]
    az = torch.arange(1024, device=DEV, dtype=torch.float32)[None, :] * (2 * math.pi / 1024)
    step = torch.arange(400, device=DEV, dtype=torch.float32)
    top = torch.tensor([nx, ny, nz], device=DEV)
    frames = []
    for f in range(case["frames"]):
        s = f / max(1, case["frames"]) * (len(line) - 1) * 0.2  # a few voxels to a scan
        i = min(int(s), len(line) - 2)
        pos = line[i] + (s - i) * (line[i + 1] - line[i])
        d = line[i + 1] - line[i]
        yaw = math.atan2(d[1], d[0])
        ray = torch.stack([el.cos() * (az + yaw).cos(), el.cos() * (az + yaw).sin(), el.sin().expand(64, 1024)], -1).view(-1, 3)
        lin = torch.zeros((ray.shape[0], 400), dtype=torch.int64, device=DEV)
        inside = torch.ones((ray.shape[0], 400), dtype=torch.bool, device=DEV)
        for k, mul in enumerate((1, nx, nx * ny)):
            v = (ray[:, k:k + 1] * step + float(pos[k]) + 0.5).floor_().to(torch.int64)
            inside &= (v >= 0) & (v < top[k])
            lin += v.clamp_(0, int(top[k]) - 1) * mul
        stop = (seen[lin] > 0) | ~inside
        end = torch.where(stop, torch.arange(400, device=DEV)[None, :], 400).amin(1)
        hit = (end < 400) & inside.gather(1, end.clamp(max=399)[:, None])[:, 0]
        passed = torch.arange(400, device=DEV)[None, :] < end[:, None]
        draws = torch.rand((3, ray.shape[0]), device=DEV, generator=g)
        # per ray, in this order: cleared voxels, the stray voxel, the hit
        clear = passed & (held[lin] > 0)
        stray = (draws[1] < 0.01) & (end > 1)
        stray_at = lin.gather(1, (draws[2] * end).long().clamp(max=399)[:, None])[:, 0]
        rays = torch.arange(ray.shape[0], device=DEV)
        cr, cs = clear.nonzero(as_tuple=True)
        order = torch.cat([cr * 512 + cs, rays[stray] * 512 + 401, rays[hit] * 512 + 402])
        where = torch.cat([lin[cr, cs], stray_at[stray], lin.gather(1, end.clamp(max=399)[:, None])[:, 0][hit]])
        value = torch.cat([torch.zeros_like(cr), torch.ones_like(stray_at[stray]), (draws[0] >= 0.01)[hit].long()])
        by = order.argsort()
        where, value = where[by], value[by]
        # the map after the frame: a voxel's last record counts
        last = torch.full((held.numel(),), -1, dtype=torch.int32, device=DEV)
        last.scatter_reduce_(0, where, torch.arange(where.numel(), device=DEV, dtype=torch.int32), "amax")
        live = last[where] == torch.arange(where.numel(), device=DEV, dtype=torch.int32)
        held[where[live]] = value[live].to(torch.uint8)
        near = torch.stack([(torch.randint(-64, 65, (65536,), device=DEV, generator=g) + int(pos[k])).clamp(0, int(top[k]) - 1)
                            for k in range(3)], 1).to(torch.int32)
        frames.append((_split(where, nx, ny).contiguous(), value.to(torch.uint8), near))
    return frames


def _trajectories(case, seed):
    """[traj, pts, 3] float32 points in metres (voxels of 0.1 m): bowed lines between points of the map."""
    g = _gen(seed + 5)
    size = torch.tensor([case["nx"], case["ny"], case["nz"]], device=DEV, dtype=torch.float32)
    a = torch.rand((case["traj"], 1, 3), device=DEV, generator=g) * (size - 2)
    b = (a + (torch.rand((case["traj"], 1, 3), device=DEV, generator=g) - 0.5) * 200).clamp_(min=0)
    bow = torch.randn((case["traj"], 1, 3), device=DEV, generator=g) * 8
    t = torch.linspace(0, 1, case["pts"], device=DEV)[None, :, None]
    p = a + t * (b - a) + (t * math.pi).sin() * bow
    return (torch.minimum(p.clamp_(min=0), size - 1) * 0.1).contiguous()


def _map(case):
    return V.Map(case["nx"], case["ny"], case["nz"], case["dmax"] or None, voxel_size=0.1)


def _ready(m, occ):
    """A map that holds `occ`, transformed."""
    m.set_occupancy_dense(occ)
    m.global_()
    m.synchronize()
    return m


def _batch_sides(case):
    """Sides of a batch's cubes, evenly over their logarithm, rounded up to a multiple of `step`."""
    lo, hi, step = math.log(case["smin"]), math.log(case["smax"]), case["step"]
    return [-(-int(math.exp(lo + (hi - lo) * (i + 0.5) / case["maps"])) // step) * step for i in range(case["maps"])]


def _batch_grids(case, seed):
    r = np.random.default_rng([int(seed), 3])
    return [_random_map(side, seed * 131 + i, r.uniform(0.01, 0.05), int(r.integers(0, 21)))
            for i, side in enumerate(_batch_sides(case))]


def _batch_records(case, seed, grids):
    out = []
    for i, o in enumerate(grids):
        g = _gen(seed * 137 + i)
        xyz = torch.randint(0, o.shape[0], (case["records"], 3), device=DEV, generator=g, dtype=torch.int32)
        out.append((xyz, torch.randint(0, 2, (case["records"],), device=DEV, generator=g, dtype=torch.uint8)))
    return out


def _dense_grid(case, seed):
    return (torch.rand((case["nz"], case["ny"], case["nx"]), device=DEV, generator=_gen(seed)) < case["p"]).to(torch.uint8)


# ---- the cases ----
def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind == "dense":
        s.update(occ=_dense_grid(case, seed), map=_map(case))
    elif kind == "noalloc":
        s.update(occ=_dense_grid(case, seed), dmax=case["dmax"])
    elif kind == "batch":
        grids = _batch_grids(case, seed)
        s.update(grids=grids, batch=V.Batch([tuple(reversed(o.shape)) for o in grids], case["dmax"]),
                 records=_batch_records(case, seed, grids))
    else:
        occ, line = _tunnel_scene(case, seed)
        m = s["map"] = _map(case)
        if kind == "tunnel":
            xyz = _coords(occ)
            s.update(xyz=xyz, val=torch.ones(xyz.shape[0], dtype=torch.uint8, device=DEV))
        elif kind == "host_masks":
            bxyz, masks = _brick_masks(occ)
            s["keep"] = [torch.from_numpy(a).pin_memory() for a in
                         (bxyz, masks.view(np.int64), _voxels(case, case["queries"], seed + 9).cpu().numpy())]
            b, k, q = (t.numpy() for t in s["keep"])
            s.update(bricks=b, masks=k.view(np.uint64), voxels=q)
        elif kind == "lidar":
            s["frames"] = _lidar_frames(case, seed, occ, line)
        elif kind == "edits":
            n = max(1, int(case["share"] * int(occ.sum())))
            g = _gen(seed + 3)
            taken = occ.view(-1).nonzero()[:, 0]
            off = taken[torch.randperm(taken.numel(), device=DEV, generator=g)[:n]]
            free = torch.randint(0, occ.numel(), (2 * n + 64,), device=DEV, generator=g)
            on = free[occ.view(-1)[free] == 0].unique()
            on = on[torch.randperm(on.numel(), device=DEV, generator=g)[:n]]
            xyz = _split(torch.cat([off, on]), case["nx"], case["ny"]).contiguous()
            val = torch.cat([torch.zeros_like(off), torch.ones_like(on)]).to(torch.uint8)
            _ready(m, occ)
            s.update(xyz=xyz, there=val, back=1 - val, graph=V.UpdateGraph(m, xyz.shape[0]),
                     voxels=_voxels(case, 1 << 16, seed + 9))
        elif kind == "points":
            _ready(m, occ)
            s.update(pts=_trajectories(case, seed), grad=torch.ones(case["traj"], device=DEV))
        else:
            _ready(m, occ)
            s["voxels"] = _voxels(case, case["queries"], seed + 9)
    return s


def _brick_masks(occ):
    """V.brick_masks of a GPU grid: coordinates [n, 3] int32 and masks [n, 8] uint64, as numpy."""
    nz, ny, nx = occ.shape
    o = torch.nn.functional.pad(occ, (0, -nx % 8, 0, -ny % 8, 0, -nz % 8))
    bz, by, bx = (d // 8 for d in o.shape)
    t = o.view(bz, 8, by, 8, bx, 8).permute(0, 2, 4, 1, 3, 5).reshape(bz, by, bx, 64, 8)
    bytes_ = (t * torch.tensor([1 << i for i in range(8)], dtype=torch.uint8, device=DEV)).sum(-1, dtype=torch.uint8)
    keep = bytes_.any(-1)
    at = keep.nonzero().flip(1).to(torch.int32).contiguous()
    return at.cpu().numpy(), bytes_[keep].contiguous().cpu().numpy().view(np.uint64)


def run(state):
    s, kind = state, state["kind"]
    if kind == "noalloc":
        return V.edt_dense_noalloc(s["occ"], s["dmax"])
    if kind == "batch":
        b = s["batch"]
        b.set_occupancy_dense(s["grids"])
        b.global_()
        for m, (xyz, val) in zip(b.maps, s["records"]):
            m.set_occupancy(xyz, val)
        b.update()
        return [m.export_dense(on_device=True) for m in b.maps]
    m = s["map"]
    if kind == "dense":
        m.set_occupancy_dense(s["occ"])
        m.global_()
        return m.export_dense(on_device=True)
    if kind == "tunnel":
        m.reset()
        m.set_occupancy(s["xyz"], s["val"])
        m.global_()
        return m.export_dense(on_device=True)
    if kind == "host_masks":
        m.reset()
        m.set_occupancy_bricks(s["bricks"], s["masks"])
        m.global_()
        return m.query(s["voxels"])
    if kind == "lidar":
        m.reset()
        seen = []
        for xyz, val, near in s["frames"]:
            m.set_occupancy(xyz, val)
            m.update()
            seen.append(m.query(near))
        return seen + [m.export_dense(on_device=True)]
    if kind == "edits":
        s["graph"].run(s["xyz"], s["there"])
        edited = m.export_dense(on_device=True)
        s["graph"].run(s["xyz"], s["back"])
        return edited, m.query(s["voxels"])
    if kind == "points":
        p = s["pts"].detach().requires_grad_(True)
        cost = V.clearance_cost(m, p, 1.0)
        cost.backward(s["grad"])
        d, g = m.distance_at(s["pts"])
        return cost.detach(), p.grad, d, g
    return m.query_nearest(s["voxels"])


def work(case):
    """Bytes of one pass (each input read once, each result written once) and a few operations per voxel and
    axis.  A tunnel scene's walls are about 3 % of its voxels; a lidar frame has about 100,000 records."""
    kind = case["kind"]
    if kind == "batch":
        vox = sum(side ** 3 for side in _batch_sides(case))
        return dict(bytes=5 * vox + 13 * case["records"] * case["maps"], flops=12 * vox)
    vox = case["nx"] * case["ny"] * case["nz"]
    if kind in ("dense", "noalloc"):
        return dict(bytes=5 * vox, flops=12 * vox)
    wall = int(0.03 * vox)
    if kind == "tunnel":
        return dict(bytes=13 * wall + 4 * vox, flops=12 * vox)
    if kind == "host_masks":
        return dict(bytes=76 * (vox // 512 // 4) + 4 * vox // 2 + 16 * case["queries"], flops=12 * vox)
    if kind == "lidar":
        return dict(bytes=case["frames"] * (13 * 100_000 + 16 * 65_536) + 4 * vox, flops=2 * vox)
    if kind == "edits":
        n = 2 * max(1, int(case["share"] * wall))
        return dict(bytes=2 * 13 * n + 16 * 65_536 + 4 * vox, flops=2 * vox)
    if kind == "points":
        n = case["traj"] * case["pts"]
        return dict(bytes=n * (3 * 12 + 12 + 16 + 8 * 4 * 3), flops=200 * n)
    return dict(bytes=case["queries"] * 24 + 8 * case["queries"], flops=100 * case["queries"])


# ---- the same in 64 bits ----
def _edt(occ, dmax):
    """Squared distance to the nearest occupied voxel by Eq. 1, one axis after the other, int64 [nz, ny, nx];
    saturated at dmax^2 (dmax 0: no truncation)."""
    reach = dmax or max(occ.shape)
    none = dmax * dmax if dmax else 1 << 40
    f = torch.where(occ > 0, 0, none)
    for axis in (2, 1, 0):
        n = f.shape[axis]
        out = f.clone()
        for d in range(1, min(reach, n)):
            a, b, src = out.narrow(axis, d, n - d), out.narrow(axis, 0, n - d), f
            torch.minimum(a, src.narrow(axis, 0, n - d) + d * d, out=a)
            torch.minimum(b, src.narrow(axis, d, n - d) + d * d, out=b)
        f = out
    return f.clamp_(max=none) if dmax else torch.where(f >= 1 << 39, 2147483647, f)


def _cell(field, pts, vs):
    """Trilinear distance at points (metres) and its gradient, in 64 bits; the cell is chosen in float32."""
    nz, ny, nx = field.shape
    u = pts / torch.tensor(vs, device=DEV, dtype=torch.float32)
    i = torch.minimum(u.floor().clamp(min=0), torch.tensor([nx - 2, ny - 2, nz - 2], device=DEV)).long()
    t = u.double() - i
    w = [torch.stack([1 - t[..., k], t[..., k]]) for k in range(3)]
    d, grad = 0.0, [0.0, 0.0, 0.0]
    for c in range(8):
        a, b, e = c & 1, c >> 1 & 1, c >> 2
        v = vs * field[i[..., 2] + e, i[..., 1] + b, i[..., 0] + a].double().sqrt()
        d = d + v * w[0][a] * w[1][b] * w[2][e]
        grad[0] = grad[0] + (2 * a - 1) * v * w[1][b] * w[2][e]
        grad[1] = grad[1] + (2 * b - 1) * v * w[0][a] * w[2][e]
        grad[2] = grad[2] + (2 * e - 1) * v * w[0][a] * w[1][b]
    return d, torch.stack(grad, -1) / vs


def exact(case, seed):
    kind = case["kind"]
    if kind in ("dense", "noalloc"):
        return _edt(_dense_grid(case, seed), case["dmax"])
    if kind not in ("tunnel", "points"):
        return None
    occ, _ = _tunnel_scene(case, seed)
    if kind == "tunnel":
        return _edt(occ, case["dmax"]) if occ.numel() <= 1 << 26 else None
    vs = float(np.float32(0.1))
    pts = _trajectories(case, seed)
    d, g = _cell(_edt(occ, case["dmax"]), pts, vs)
    h = (1.0 - d).clamp(min=0)
    return h.square().sum(1), -2 * h[..., None] * g, d, g
