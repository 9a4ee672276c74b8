"""Device memory at its limits: a server's budget holds as many requests in flight as their depth buffers and
the step counts of their largest levels allow, whatever else their counts could use; and an allocator that has
refused a large workspace is not asked for it again by every later call."""
import math
import threading
import time

import numpy as np
import pytest

import synth
from synth import Sensor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2609_40297_gb300 as mig  # noqa: E402


def _problem(seed, sensor, n=24, depth=6):
    return synth.random_small(seed, nx=60, ny=60, nz=30, v=0.1, p_occ=0.001, n_nodes=n, max_depth=depth, sensor=sensor)


def _bytes(parent, s, counts, columns):
    """Depth buffers, plan, counters (also per column) and, with counts, a uint16 per ray of the largest level."""
    parent = np.asarray(parent)
    depth = np.zeros(len(parent), int)
    for i in range(len(parent)):
        j = parent[i]
        while j >= 0:
            depth[i] += 1
            j = parent[j]
    n, levels, rays, K = len(parent), depth.max() + 1, s.width * s.height, s.yaw_bins
    parts = [16 * n, 8 * n, 4 * max(1, depth.sum()), 4 * (levels + 1), 4 * levels, 4 * n, 8 * n * K, 4 * levels, 12 * n, 4 * n,
             4 * max(1, len(set(parent[parent >= 0]))) * rays]
    if counts:
        parts += [2 * np.bincount(depth).max() * K * rays, 256]
    if columns:
        parts += [8 * n * K * math.ceil(s.width * 360 / (s.hfov_deg * K))]
    return int(sum((p + 255) // 256 * 256 for p in parts))


@pytest.mark.parametrize("mode", [mig.MODE_MARGINAL, mig.MODE_ABSOLUTE, mig.MODE_INTERVAL, mig.MODE_PANORAMIC])
@pytest.mark.parametrize("image", [(40, 30, 8), (9, 6, 3), (96, 72, 2)])
def test_budget_holds_its_requests(image, mode):
    w, h, yaws = image
    p = _problem(141, Sensor(90, 60, w, h, 2.0, yaws, 0.0))
    busy = _problem(142, Sensor(90, 60, 320, 240, 2.0, 36, 0.0), 600, 12)
    counts = mode in (mig.MODE_MARGINAL, mig.MODE_ABSOLUTE)
    flight = 5
    budget = flight * _bytes(p.tree.parent, p.sensor, counts, mode == mig.MODE_PANORAMIC)
    ctx = mig.Context(0, stream=torch.cuda.Stream())
    m = mig.Map(ctx, p.map.grid, p.map.voxel_size, p.map.origin)
    try:
        want = mig.tree_eval(m, p.tree.parent, p.tree.pos, p.sensor, mode=mode)
        peaks = []
        for k in (1, flight):
            srv = mig.Server(ctx, arena_budget_bytes=budget, max_inflight=4096)
            try:
                # a long call holds the context until all requests wait, so that they are admitted together
                holds = threading.Thread(target=mig.tree_eval_stats, args=(m, busy.tree.parent, busy.tree.pos, busy.sensor))
                holds.start()
                time.sleep(0.02)
                subs = [srv.submit(m, p.tree.parent, p.tree.pos, p.sensor, mode=mode) for _ in range(k)]
                assert holds.is_alive()
                for t, _ in subs:
                    assert srv.poll(t, timeout_us=30_000_000)
                holds.join()
                peaks.append(srv.memory()["peak"])
                for _, got in subs:
                    for key in ("abs", "marg", "yaw"):
                        assert np.array_equal(got[key], want[key]), key
            finally:
                srv.close()
        assert peaks[1] == flight * peaks[0] and peaks[1] <= budget
    finally:
        m.close()
        ctx.close()


@pytest.mark.parametrize("call", ["host", "device", "batch", "server"])
def test_refused_memory_is_not_asked_for_by_every_call(monkeypatch, call):
    """An allocator with a limit below the largest workspace: the first call finds the one that fits, the next
    ones ask for no more than that (calls whose memory is kept: for nothing), with the same results."""
    limit, asked = [1 << 62], []
    real = mig._torch_allocator

    def limited(device):
        a = real(device)

        def alloc(nbytes, stream, user):
            asked.append(int(nbytes))
            return None if nbytes > limit[0] else a.alloc(nbytes, stream, user)

        b = mig.Allocator(mig.ALLOC_FN(alloc), a.free, None)
        b.keep = (a, alloc)
        return b

    monkeypatch.setattr(mig, "_torch_allocator", limited)
    p = _problem(143, Sensor(90, 60, 40, 30, 2.0, 8, 0.0))
    c = mig.Context(0, stream=torch.cuda.Stream())
    m = mig.Map(c, p.map.grid, p.map.voxel_size, p.map.origin)
    srv = mig.Server(c, arena_budget_bytes=1 << 30, max_inflight=2) if call == "server" else None
    par, pos = torch.from_numpy(p.tree.parent).cuda(), torch.from_numpy(p.tree.pos).cuda()
    out = [torch.empty(p.tree.n, dtype=torch.int32, device="cuda") for _ in range(3)]

    def run():
        if call == "device":
            mig.tree_eval_device(m, par, pos, p.sensor, 6, *out)
            c.sync()
            return [t.cpu().numpy() for t in out]
        if call == "batch":
            got = mig.tree_eval_batch(c, [(p.tree.parent, p.tree.pos, p.sensor)] * 2, [m, m])[1]
        elif call == "server":
            ticket, got = srv.submit(m, p.tree.parent, p.tree.pos, p.sensor)
            assert srv.poll(ticket, timeout_us=30_000_000)
        else:
            got = mig.tree_eval(m, p.tree.parent, p.tree.pos, p.sensor)
        return [got[k] for k in ("abs", "marg", "yaw")]

    try:
        mig.tree_eval(m, p.tree.parent[:1], p.tree.pos[:1], p.sensor)  # the camera's tables and a small workspace
        asked.clear()
        limit[0] = (1 << 20) if call == "batch" else (1 << 19)  # no room for any step counts beside the queue
        first = run()
        assert any(b > limit[0] for b in asked)
        for i in range(20):
            asked.clear()
            assert all(np.array_equal(a, b) for a, b in zip(run(), first))
            assert all(b <= limit[0] for b in asked), (i, asked)
            assert call == "server" or not asked
    finally:
        limit[0] = 1 << 62
        if srv is not None:
            srv.close()
        m.close()
        c.close()


def test_request_is_retried_once_memory_is_there(monkeypatch):
    """A request that needs the least it can and is refused fails; the next one like it is asked for again."""
    limit = [1 << 62]
    real = mig._torch_allocator

    def limited(device):
        a = real(device)

        def alloc(nbytes, stream, user):
            return None if nbytes > limit[0] else a.alloc(nbytes, stream, user)

        b = mig.Allocator(mig.ALLOC_FN(alloc), a.free, None)
        b.keep = (a, alloc)
        return b

    monkeypatch.setattr(mig, "_torch_allocator", limited)
    p = _problem(144, Sensor(90, 60, 40, 30, 2.0, 8, 0.0))
    c = mig.Context(0, stream=torch.cuda.Stream())
    m = mig.Map(c, p.map.grid, p.map.voxel_size, p.map.origin)
    srv = mig.Server(c, arena_budget_bytes=1 << 30, max_inflight=2)
    try:
        want = mig.tree_eval(m, p.tree.parent, p.tree.pos, p.sensor)
        for kernel in (mig.COUNT_RAYS, mig.COUNT_AUTO):  # without a region for the counts, and with one
            c.set_count_kernel(kernel, 0)
            limit[0] = 1 << 14
            t, _ = srv.submit(m, p.tree.parent, p.tree.pos, p.sensor)
            with pytest.raises(mig.MigError) as e:
                srv.poll(t, timeout_us=30_000_000)
            assert e.value.status == mig.MIG_ENOMEM
            limit[0] = 1 << 62
            for _ in range(2):
                t, got = srv.submit(m, p.tree.parent, p.tree.pos, p.sensor)
                assert srv.poll(t, timeout_us=30_000_000)
                for k in ("abs", "marg", "yaw"):
                    assert np.array_equal(got[k], want[k]), k
    finally:
        limit[0] = 1 << 62
        srv.close()
        m.close()
        c.close()


def test_step_budget_holds_in_small_regions():
    """A request between its level's step counts and the queue's least size takes whole nodes into what its share
    leaves, but no more of them than the context's budget of step counts."""
    p = _problem(145, Sensor(90, 60, 40, 30, 2.0, 8, 0.0))
    bare = _bytes(p.tree.parent, p.sensor, False, False)
    node = 2 * 8 * 40 * 30
    peaks = {}
    for nodes in (1, 3, 1000):
        ctx = mig.Context(0, stream=torch.cuda.Stream())
        m = mig.Map(ctx, p.map.grid, p.map.voxel_size, p.map.origin)
        want = mig.tree_eval(m, p.tree.parent, p.tree.pos, p.sensor)
        ctx.set_count_kernel(mig.COUNT_NODES, nodes * node + 100)
        srv = mig.Server(ctx, arena_budget_bytes=bare + (2 << 20), max_inflight=1)
        try:
            t, got = srv.submit(m, p.tree.parent, p.tree.pos, p.sensor)
            assert srv.poll(t, timeout_us=30_000_000)
            peaks[nodes] = srv.memory()["peak"]
            for k in ("abs", "marg", "yaw"):
                assert np.array_equal(got[k], want[k]), k
        finally:
            srv.close()
            m.close()
            ctx.close()
    assert bare + node < peaks[1] <= peaks[3] - 2 * node and peaks[3] <= peaks[1000] - node
    assert peaks[1000] <= bare + (2 << 20)
