"""The per-node count by 4x4x4 bricks against the ray-by-ray count kernels on the same inputs, bit for
bit, where the bricks, macro blocks, tile bounds and queue have their edges: grids whose sides are no
multiple of 4, 16 or 8 voxels, ranges below one brick, images of a few pixels and with partial tiles,
more yaws than one record holds, deep trees, positions on brick faces, wide and steep cameras. Also the
map's brick data under updates, and the allocation-free call where its scratch holds few nodes."""
import numpy as np
import pytest

import synth
from synth import Sensor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2609_40297_gb300 as mig  # noqa: E402

KEYS = ("abs", "marg", "yaw", "cnt_abs", "cnt_marg", "depth")
MODES = {"marginal": mig.MODE_MARGINAL, "single_parent": mig.MODE_SINGLE_PARENT, "interval": mig.MODE_INTERVAL}
# (grid, voxel, occupied share, nodes, depth, sensor)
CASES = [
    ((24, 20, 12), 0.25, 0.08, 12, 5, Sensor(80, 55, 19, 13, 2.5, 6, 0.0)),
    ((33, 29, 17), 0.25, 0.02, 16, 6, Sensor(90, 60, 36, 24, 4.0, 8, 0.0)),
    ((65, 47, 30), 0.2, 0.004, 20, 12, Sensor(87, 58, 48, 28, 5.0, 16, 10.0)),
    ((61, 66, 23), 0.2, 0.01, 14, 4, Sensor(90, 60, 33, 17, 6.0, 70, 0.0)),
    ((30, 31, 14), 0.25, 0.05, 10, 4, Sensor(120, 90, 7, 5, 3.0, 3, -20.0)),
    ((30, 31, 14), 0.25, 0.05, 10, 4, Sensor(60, 40, 9, 8, 0.6, 5, 0.0)),
    ((40, 37, 25), 0.25, 0.02, 12, 5, Sensor(170, 150, 41, 35, 4.0, 9, 35.0)),
    ((40, 37, 25), 0.25, 0.02, 12, 5, Sensor(30, 20, 130, 70, 5.0, 12, -70.0)),
    ((130, 100, 40), 0.1, 0.0005, 24, 20, Sensor(90, 60, 64, 48, 6.0, 12, 5.0)),
]


def _eval(ctx, m, p, mode, kernel):
    ctx.set_count_kernel(kernel, 0)
    try:
        return mig.tree_eval(m, p.tree.parent, p.tree.pos, p.sensor, mode=mode, want_counts=True, want_depth=True)
    finally:
        ctx.set_count_kernel(mig.COUNT_AUTO, 0)


def _same(a, b, what):
    for k in KEYS:
        assert np.array_equal(a[k], b[k]), (what, k, np.argwhere(a[k] != b[k])[:4].tolist())


@pytest.fixture(scope="module")
def ctx():
    c = mig.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("mode", sorted(MODES))
@pytest.mark.parametrize("ci", range(len(CASES)))
def test_bricks_equal_rays(ctx, ci, mode):
    (nx, ny, nz), v, occ, nodes, depth, sensor = CASES[ci]
    p = synth.random_small(800 + ci, nx=nx, ny=ny, nz=nz, v=v, p_occ=occ, n_nodes=nodes, max_depth=depth, sensor=sensor)
    p.tree.pos[1::2] = np.round(p.tree.pos[1::2] / v) * v  # every second node on voxel corners
    p.tree.pos = np.clip(p.tree.pos, 0, (np.array([nx, ny, nz]) - 0.5) * v).astype(np.float32)
    m = mig.Map(ctx, p.map.grid, v, p.map.origin)
    try:
        rays = _eval(ctx, m, p, MODES[mode], mig.COUNT_RAYS)
        assert rays["abs"].sum() > 0
        _same(_eval(ctx, m, p, MODES[mode], mig.COUNT_NODES), rays, (ci, mode))
    finally:
        m.close()


# few and many columns per brick, one row, one to 70 yaws, a node's brick around the seam
PANO = CASES[:3] + CASES[5:] + [
    ((30, 31, 14), 0.25, 0.05, 10, 4, Sensor(179, 60, 1, 1, 3.0, 1, 0.0)),
    ((40, 37, 25), 0.2, 0.02, 12, 5, Sensor(20, 130, 90, 3, 5.0, 70, 0.0)),
    ((67, 61, 30), 0.1, 0.003, 16, 6, Sensor(10, 60, 640, 40, 4.0, 16, 0.0)),
    ((67, 61, 30), 0.1, 0.003, 30, 2, Sensor(87, 58, 100, 75, 5.0, 5, 0.0)),
]


@pytest.mark.parametrize("budget", [0, 1 << 18])
@pytest.mark.parametrize("ci", range(len(PANO)))
def test_panoramic_bricks_equal_rays(ctx, ci, budget):
    """The panoramic mode, with the whole level and with few nodes at a time (or none: ray by ray)."""
    (nx, ny, nz), v, occ, nodes, depth, s = PANO[ci]
    sensor = Sensor(s.hfov_deg, s.vfov_deg, s.width, s.height, s.range_m, s.yaw_bins, 0.0)
    p = synth.random_small(850 + ci, nx=nx, ny=ny, nz=nz, v=v, p_occ=occ, n_nodes=nodes, max_depth=depth, sensor=sensor)
    p.tree.pos[1::2] = np.round(p.tree.pos[1::2] / v) * v  # every second node on voxel corners
    p.tree.pos[2::4] = (np.floor(p.tree.pos[2::4] / v) + 0.5) * v  # and every fourth on a voxel centre
    p.tree.pos = np.clip(p.tree.pos, 0, (np.array([nx, ny, nz]) - 0.5) * v).astype(np.float32)
    m = mig.Map(ctx, p.map.grid, v, p.map.origin)
    try:
        rays = _eval(ctx, m, p, mig.MODE_PANORAMIC, mig.COUNT_RAYS)
        assert rays["abs"].sum() > 0
        ctx.set_count_kernel(mig.COUNT_NODES, budget)
        try:
            got = mig.tree_eval(m, p.tree.parent, p.tree.pos, p.sensor, mode=mig.MODE_PANORAMIC, want_counts=True,
                                want_depth=True)
        finally:
            ctx.set_count_kernel(mig.COUNT_AUTO, 0)
        _same(got, rays, ci)
    finally:
        m.close()


@pytest.mark.parametrize("mode", ["marginal", "interval"])
def test_brick_data_follows_updates(ctx, mode):
    """Boxes of unknown, free and occupied voxels written over a sparse map whose sides are no multiple
    of 4: masks and distances equal those of a map made afresh, seen through the results."""
    rng = np.random.default_rng(3)
    p = synth.random_small(31, nx=101, ny=90, nz=38, v=0.1, p_occ=0.0003, n_nodes=14, max_depth=5,
                           sensor=Sensor(90, 60, 48, 36, 5.0, 8, 0.0))
    g = p.map.grid.copy()
    m = mig.Map(ctx, g, p.map.voxel_size, p.map.origin)
    try:
        for i in range(5):
            d = rng.integers(1, [30, 30, 20])
            x, y, z = (int(rng.integers(0, s - e + 1)) for s, e in zip((101, 90, 38), d))
            box = rng.choice(np.array([0, 1, 2], np.uint8), size=tuple(d[::-1]), p=[[0.5, 0.5, 0], [0.4, 0.5, 0.1]][i % 2])
            m.update(x, y, z, box)
            g[z:z + d[2], y:y + d[1], x:x + d[0]] = box
            fresh = mig.Map(ctx, g, p.map.voxel_size, p.map.origin)
            try:
                _same(_eval(ctx, m, p, MODES[mode], mig.COUNT_NODES), _eval(ctx, fresh, p, MODES[mode], mig.COUNT_RAYS), i)
            finally:
                fresh.close()
    finally:
        m.close()


@pytest.mark.parametrize("width,height,yaws", [(160, 120, 16), (640, 480, 3), (1024, 700, 2), (24, 18, 200)])
def test_noalloc_chunks(ctx, width, height, yaws):
    """The fixed scratch from room for many nodes at a time down to none (counted ray by ray)."""
    p = synth.random_small(55, nx=60, ny=60, nz=30, v=0.1, p_occ=0.001, n_nodes=18, max_depth=6,
                           sensor=Sensor(90, 60, width, height, 2.5, yaws, 10.0))
    m = mig.Map(ctx, p.map.grid, p.map.voxel_size, p.map.origin)
    dev = torch.device("cuda:0")
    try:
        par, pos = torch.from_numpy(p.tree.parent).to(dev), torch.from_numpy(p.tree.pos).to(dev)
        outs = []
        for call in (mig.tree_eval_device, mig.tree_eval_device_noalloc):
            o = [torch.full((p.tree.n,), -7, dtype=torch.int32, device=dev) for _ in range(3)]
            call(m, par, pos, p.sensor, 6, *o)
            ctx.sync()
            outs.append([t.cpu().numpy() for t in o])
        rays = _eval(ctx, m, p, mig.MODE_MARGINAL, mig.COUNT_RAYS)
        for a, b, k in zip(*outs, ("abs", "marg", "yaw")):
            assert np.array_equal(a, b) and np.array_equal(a, rays[k]), k
    finally:
        m.close()


@pytest.mark.parametrize("call", ["host", "panoramic", "interval", "device", "batch"])
def test_less_memory(monkeypatch, call):
    """An allocator that refuses the largest request: the tree's step counts, then the level's, then none
    (ray by ray), with the same results."""
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
    p = synth.random_small(77, nx=60, ny=60, nz=30, v=0.1, p_occ=0.001, n_nodes=24, max_depth=6,
                           sensor=Sensor(90, 60, 40, 30, 2.0, 8, 0.0))

    def run(most):
        c = mig.Context(0)
        try:
            m = mig.Map(c, p.map.grid, p.map.voxel_size, p.map.origin)
            try:
                if call == "panoramic":  # the camera's tables
                    mig.tree_eval(m, p.tree.parent[:1], p.tree.pos[:1], p.sensor, mode=mig.MODE_PANORAMIC)
                limit[0] = most
                asked.clear()
                if call == "device":
                    par, pos = torch.from_numpy(p.tree.parent).cuda(), torch.from_numpy(p.tree.pos).cuda()
                    o = [torch.empty(p.tree.n, dtype=torch.int32, device="cuda") for _ in range(3)]
                    mig.tree_eval_device(m, par, pos, p.sensor, 6, *o)
                    c.sync()
                    return [t.cpu().numpy() for t in o]
                if call == "batch":
                    got = mig.tree_eval_batch(c, [(p.tree.parent, p.tree.pos, p.sensor)] * 2, [m, m])[1]
                else:
                    got = mig.tree_eval(m, p.tree.parent, p.tree.pos, p.sensor, mode=MODES.get(call, mig.MODE_MARGINAL)
                                        if call != "panoramic" else mig.MODE_PANORAMIC)
                return [got[k] for k in ("abs", "marg", "yaw")]
            finally:
                limit[0] = 1 << 62
                m.close()
        finally:
            c.close()

    want, steps, most = run(1 << 62), 0, 1 << 62
    while True:
        need = [b for b in asked if b <= most]
        most = max(need) - 1
        try:
            got = run(most)
        except mig.MigError:
            break
        steps += 1
        assert all(np.array_equal(a, b) for a, b in zip(got, want)), steps
    # the device call does not know its levels' sizes: there the level's step counts are the tree's
    assert steps >= (1 if call == "device" else 2)


@pytest.mark.parametrize("call", ["marginal", "interval", "panoramic", "device", "noalloc"])
@pytest.mark.parametrize("width,height", [(6, 4), (160, 120)])
def test_coarse_images_are_walked(ctx, call, width, height):
    """An image whose pixels lie farther apart than the voxels over most of the range (the default counts it
    ray by ray) and a fine one: equal to the count by voxels."""
    p = synth.random_small(91, nx=130, ny=120, nz=50, v=0.1, p_occ=0.0003, n_nodes=200, max_depth=2,
                           sensor=Sensor(90, 60, width, height, 9.0, 16 if width < 10 else 2, 0.0))
    m = mig.Map(ctx, p.map.grid, p.map.voxel_size, p.map.origin)
    dev = torch.device("cuda:0")
    par, pos = torch.from_numpy(p.tree.parent).to(dev), torch.from_numpy(p.tree.pos).to(dev)
    try:
        outs = []
        for kernel in (mig.COUNT_AUTO, mig.COUNT_NODES):
            if call in ("device", "noalloc"):
                ctx.set_count_kernel(kernel, 0)
                o = [torch.full((p.tree.n,), -7, dtype=torch.int32, device=dev) for _ in range(3)]
                try:
                    (mig.tree_eval_device if call == "device" else mig.tree_eval_device_noalloc)(m, par, pos, p.sensor, 2, *o)
                    ctx.sync()
                finally:
                    ctx.set_count_kernel(mig.COUNT_AUTO, 0)
                outs.append(dict(zip(("abs", "marg", "yaw"), [t.cpu().numpy() for t in o])))
            else:
                outs.append(_eval(ctx, m, p, MODES.get(call, mig.MODE_PANORAMIC), kernel))
        assert outs[0]["abs"].sum() > 0
        for k in outs[0]:
            if isinstance(outs[0][k], np.ndarray):
                assert np.array_equal(outs[0][k], outs[1][k]), k
        if call == "marginal":
            st = mig.tree_eval_stats(m, p.tree.parent, p.tree.pos, p.sensor)[1]
            assert st["voxel_pass"] == (mig.COUNT_RAYS if width < 10 else mig.COUNT_NODES)
    finally:
        m.close()
