"""Ordering between the caller's current torch stream and the map's own: inputs still being produced when the
call is made, and results used right after it, from a side stream, the default stream and two threads."""
import threading

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


def session(V, torch, seed, out):
    rs = np.random.default_rng(seed)
    side = torch.cuda.Stream()
    m = V.Map(40, 33, 27, 9)
    occ = np.zeros((27, 33, 40), np.uint8)
    ok = True
    for frame in range(6):
        xyz = np.stack([rs.integers(0, n, 30) for n in (40, 33, 27)], 1).astype(np.int32)
        val = rs.integers(0, 2, 30).astype(np.uint8)
        for (x, y, z), v in zip(xyz, val):
            occ[z, y, x] = v
        host = torch.from_numpy(xyz).pin_memory(), torch.from_numpy(val).pin_memory()
        with torch.cuda.stream(side if frame % 2 else torch.cuda.default_stream()):
            a, b = torch.zeros((30, 3), dtype=torch.int32, device="cuda"), torch.zeros(30, dtype=torch.uint8, device="cuda")
            torch.cuda._sleep(2_000_000)  # about a millisecond: the call below is made before the inputs are there
            a.copy_(host[0], non_blocking=True)
            b.copy_(host[1], non_blocking=True)
            m.set_occupancy(a, b)
            m.update()
            d = m.export_dense(on_device=True)
            total = d.sum()  # ordered behind the export by the call itself
            torch.cuda.current_stream().synchronize()
            ref = O.edt_factorised(occ, 9)
            ok &= bool(np.array_equal(d.cpu().numpy(), ref)) and int(total) == int(ref.sum())
    m.close()
    out.append(ok)


def test_caller_streams():
    import torch
    import paper_2105_04419_gb300 as V
    out = []
    threads = [threading.Thread(target=session, args=(V, torch, s, out)) for s in (1, 2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    session(V, torch, 3, out)
    assert out == [True, True, True]


@pytest.mark.parametrize("pinned", [False, True])
def test_host_queries_behind_a_running_transform(pinned):
    import torch
    import paper_2105_04419_gb300 as V
    rs = np.random.default_rng(5)
    occ = (rs.random((64, 90, 130)) < 0.001).astype(np.uint8)
    m = V.Map(130, 90, 64, 20)
    grid = torch.from_numpy(occ).cuda()
    for n in (1, 1000, 300000, 17):  # the buffer grows, then is larger than the call
        m.set_occupancy_dense(grid)
        m.global_()
        q = torch.from_numpy(np.stack([rs.integers(-1, k + 1, n) for k in (130, 90, 64)], 1).astype(np.int32))
        q = (q.pin_memory() if pinned else q).numpy()
        ref = np.pad(O.edt_factorised(occ, 20), 1, constant_values=400)
        assert np.array_equal(m.query(q), ref[q[:, 2] + 1, q[:, 1] + 1, q[:, 0] + 1])
        grid = torch.from_numpy(np.ascontiguousarray(occ[::-1])).cuda()
        occ = np.ascontiguousarray(occ[::-1])
    m.close()


@pytest.mark.parametrize("call", ["query", "query_nearest", "set_occupancy"])
@pytest.mark.parametrize("joined", [False, True])
def test_host_arrays_are_read_in_the_stream_s_order(call, joined):
    """A page-locked array that a copy still queued on the map's stream (or on one it was made to wait for) fills."""
    import torch
    import paper_2105_04419_gb300 as V
    from paper_2105_04419_gb300 import lib as L
    rs = np.random.default_rng(7)
    occ = (rs.random((64, 90, 130)) < 0.001).astype(np.uint8)
    own, side = torch.cuda.Stream(), torch.cuda.Stream()
    m = V.Map(130, 90, 64, 20, stream=own)
    for n in (1, 1000, 200000):
        m.set_occupancy_dense(occ)
        m.global_()
        xyz = np.stack([rs.integers(0, k, n) for k in (130, 90, 64)], 1).astype(np.int32)
        there = torch.from_numpy(xyz).cuda()
        pinned = torch.zeros((n, 3), dtype=torch.int32).pin_memory()
        one = torch.ones(n, dtype=torch.uint8).pin_memory().numpy()
        want = getattr(m, call)(xyz) if call != "set_occupancy" else None
        if call == "query":
            m.query(pinned.numpy())  # the buffers are there: nothing in the call below waits for an allocation
        torch.cuda.synchronize()
        with torch.cuda.stream(side if joined else own):
            torch.cuda._sleep(20_000_000)  # about ten milliseconds
            pinned.copy_(there, non_blocking=True)
            if joined:
                assert L.load().vdbedt_wait_stream(m.handle, side.cuda_stream) == 0
            if call == "set_occupancy":
                m.set_occupancy(pinned.numpy(), one)
            else:
                assert np.array_equal(getattr(m, call)(pinned.numpy()), want), n
        if call == "set_occupancy":
            m.update()
            now = occ.copy()
            now[xyz[:, 2], xyz[:, 1], xyz[:, 0]] = 1
            assert np.array_equal(m.export_dense(), O.edt_factorised(now, 20)), n
    m.close()


@pytest.mark.parametrize("captured", ["map", "caller"])
def test_a_refused_stream_order_leaves_the_map_usable(captured):
    """A call from a stream outside the capture of the map's own (or the reverse) is refused; later calls answer."""
    import ctypes
    import torch
    import paper_2105_04419_gb300 as V
    from paper_2105_04419_gb300 import lib as L
    rt = ctypes.CDLL("libcudart.so.13")
    occ = (np.random.default_rng(3).random((20, 30, 40)) < 0.01).astype(np.uint8)
    side = torch.cuda.Stream()
    m = V.Map(40, 30, 20, 8)
    m.set_occupancy_dense(occ)
    m.global_()
    q = torch.zeros((5, 3), dtype=torch.int32, device="cuda")
    want = m.query(q).cpu()
    torch.cuda.synchronize()
    stream = ctypes.c_void_p((m.stream if captured == "map" else side).cuda_stream)
    graph = ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(stream, 2) == 0  # relaxed
    try:
        if captured == "map":
            with pytest.raises(RuntimeError):
                m.query(q)
        else:
            assert L.load().vdbedt_join_stream(m.handle, side.cuda_stream) != 0
    finally:
        rt.cudaStreamEndCapture(stream, ctypes.byref(graph))
        rt.cudaGetLastError()
        if graph:
            rt.cudaGraphDestroy(graph)
    assert torch.equal(m.query(q).cpu(), want)
    assert np.array_equal(m.export_dense(), O.edt_factorised(occ, 8))
    m.close()


def test_calls_inside_a_caller_s_own_capture():
    """A caller's graph on a stream that is not the map's: the map's first kernel after each join follows a kernel, a copy
    or nothing of the caller's, and a second stream joins between.  Replays answer as eager calls on another map."""
    import torch
    import paper_2105_04419_gb300 as V
    rs = np.random.default_rng(11)
    nx, ny, nz, n = 130, 90, 64, 400
    occ = torch.from_numpy((rs.random((nz, ny, nx)) < 0.001).astype(np.uint8)).cuda()
    maps = [V.Map(nx, ny, nz, 20) for _ in range(2)]
    buf = torch.zeros((n, 3), dtype=torch.int32, device="cuda")
    val = torch.zeros(n, dtype=torch.uint8, device="cuda")

    def session(m):
        cur, other = torch.cuda.current_stream(), torch.cuda.Stream()
        out = [m.query(buf)]                            # nothing of the caller's before it
        z = torch.empty_like(occ)
        z.copy_(occ)                                    # a copy
        m.set_occupancy_dense(z)
        m.global_()
        m.set_occupancy(buf + 0, val + 0)               # kernels
        m.update()
        out.append(m.query(buf + 0) * 2)
        other.wait_stream(cur)
        with torch.cuda.stream(other):
            x = torch.clamp(buf + 1, max=nz - 1)
            m.set_occupancy(x, 1 - val)
            m.update()
            near = m.query_nearest(x)
        cur.wait_stream(other)
        d, g = m.distance_at((x.float() * 0.1).contiguous())
        return out + [near, d, g, m.export_dense(on_device=True)]

    stream = torch.cuda.Stream()
    for m in maps:
        m.set_occupancy_dense(occ)
        m.global_()
        with torch.cuda.stream(stream):
            session(m)
        torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        got = session(maps[0])
    for _ in range(8):
        buf.copy_(torch.from_numpy(np.stack([rs.integers(0, k, n) for k in (nx, ny, nz)], 1).astype(np.int32)))
        val.copy_(torch.from_numpy(rs.integers(0, 2, n).astype(np.uint8)))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        want = session(maps[1])
        torch.cuda.synchronize()
        assert [torch.equal(a, b) for a, b in zip(got, want)] == [True] * len(want)
    del graph
    for m in maps:
        m.close()
