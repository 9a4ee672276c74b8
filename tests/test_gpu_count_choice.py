"""Which way a tree is counted by default, and both ways where only one is the default: short ranges with
fine images, ranges far beyond the grid and coarse images (the pass that ran is in the statistics); the
longest range (1024 voxels) ray by ray and by voxels; and a queue of undecided bricks that overflows."""
import ctypes as C
import math

import numpy as np
import pytest

import synth
from synth import Sensor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2609_40297_gb300 as mig  # noqa: E402
from test_gpu_parity import assert_same, run_both  # noqa: E402

MODES = (mig.MODE_MARGINAL, mig.MODE_SINGLE_PARENT, mig.MODE_ABSOLUTE, mig.MODE_INTERVAL, mig.MODE_PANORAMIC)


@pytest.fixture(scope="module")
def ctx():
    c = mig.Context(0)
    yield c
    c.close()


def _tree(rng, n, dims, v, spread):
    mid = np.array(dims) / 2.0
    pos = ((mid + rng.uniform(-spread, spread, (n, 3))) * v).astype(np.float32)
    parent = np.array([-1] + [(i - 1) // 2 for i in range(1, n)], np.int32)  # a binary tree
    return parent, pos


@pytest.mark.parametrize("dims,v,sensor,nodes,want", [
    ((64, 64, 32), 0.05, Sensor(60, 68, 39, 25, 5.4, 25, 0.0), 300, mig.COUNT_NODES),   # a range beyond the grid
    ((64, 64, 32), 0.2, Sensor(90, 60, 240, 160, 1.0, 16, 0.0), 200, mig.COUNT_NODES),  # 5 voxels of range
    ((200, 200, 50), 0.2, Sensor(90, 60, 160, 120, 5.0, 16, 0.0), 100, mig.COUNT_NODES),
    ((400, 400, 100), 0.05, Sensor(90, 60, 20, 14, 7.5, 16, 0.0), 300, mig.COUNT_RAYS),  # coarse, long
])
def test_default_pass(ctx, dims, v, sensor, nodes, want):
    rng = np.random.default_rng(5)
    grid = np.where(rng.random(dims[::-1]) < 0.002, 2, 0).astype(np.uint8)
    parent, pos = _tree(rng, nodes, dims, v, min(dims) / 4)
    m = mig.Map(ctx, grid, v)
    try:
        assert mig.tree_eval_stats(m, parent, pos, sensor)[1]["voxel_pass"] == want
    finally:
        m.close()


@pytest.mark.parametrize("writes", ["whole", "one box", "one voxel", "voxel by voxel"])
def test_allocation_free_choice_of_a_map_written_in_parts(ctx, writes):
    """A few occupied voxels in an empty map are no clutter, however they came there: the allocation-free call
    counts fine images over 20 voxels of range by voxels."""
    dims, v, n = (64, 64, 32), 0.1, 30
    rng = np.random.default_rng(11)
    parent, pos = _tree(rng, n, dims, v, 8)
    sensor = Sensor(90, 60, 160, 120, 2.0, 8, 0.0)
    grid = np.zeros(dims[::-1], np.uint8)
    at = rng.integers(0, 32, (1 if writes == "one voxel" else 20, 3))
    grid[at[:, 0], at[:, 1], at[:, 2]] = 2
    m = mig.Map(ctx, grid if writes == "whole" else np.zeros_like(grid), v)
    if writes != "whole":  # a map created without voxels, through the C call
        m.close()
        m.h = C.c_void_p()
        mig.check(mig.lib().mig_map_create(ctx.h, *dims, v, (C.c_float * 3)(), None, C.byref(m.h)))
    dev = torch.device("cuda:0")
    try:
        if writes == "one box":
            m.update(0, 0, 0, np.ascontiguousarray(grid[:, :32, :32]))
        elif writes != "whole":
            for z, y, x in at:
                m.update(int(x), int(y), int(z), np.full((1, 1, 1), 2, np.uint8))
        assert np.array_equal(m.read(), grid)
        par, p = torch.from_numpy(parent).to(dev), torch.from_numpy(pos).to(dev)
        out = [torch.empty(n, dtype=torch.int32, device=dev) for _ in range(3)]
        ctx.profile(True)
        ctx.profile_read()
        mig.tree_eval_device_noalloc(m, par, p, sensor, 4, *out)
        ctx.sync()
        t = ctx.profile_read()
        assert t["cast_launches"] > 0 and t["count_launches"] == 0
    finally:
        ctx.profile(False)
        m.close()


@pytest.mark.parametrize("kernel", [mig.COUNT_RAYS, mig.COUNT_NODES, mig.COUNT_PAIRS])
def test_longest_range_by_each_kernel(ctx, kernel):
    """The 4096-voxel axis and 1024-voxel range of the limit tests, by each count kernel."""
    rng = np.random.default_rng(94)
    v = 0.05
    grid = np.where(rng.random((7, 9, 4096)) < 0.5, 0, 1).astype(np.uint8)
    grid[:, :, 3900:] = 2
    grid[2:5, :, 2500:2503] = 2
    xs = np.array([100.3, 610.7, 1500.1, 2100.9, 2495.2])
    pos = (np.stack([xs, np.full(5, 4.4), np.full(5, 3.3)], 1) * v).astype(np.float32)
    parent = np.array([-1, 0, 1, 2, 3], np.int32)
    s = Sensor(30, 30, 9, 7, 1024 * v, 2, 0.0)
    ctx.set_count_kernel(kernel, 0)
    try:
        for mode in MODES:
            got, ref = run_both(ctx, grid, v, (0, 0, 0), parent, pos, s, mode=mode, depth=(mode == mig.MODE_MARGINAL))
            assert_same(got, ref)
            assert got["abs"].sum() > 0
    finally:
        ctx.set_count_kernel(mig.COUNT_AUTO, 0)


@pytest.mark.parametrize("mode,yaws", [(mig.MODE_MARGINAL, 8), (mig.MODE_MARGINAL, 70), (mig.MODE_INTERVAL, 70),
                                       (mig.MODE_PANORAMIC, 8)])
def test_queue_overflow(ctx, mode, yaws):
    """An unknown map and a coarse, wide camera leave nearly every brick of the range ball undecided, more
    than the queue holds (at least 2^16 and 0.3 to 0.7 of an upper bound of the ball's bricks, per node): the
    last ones are counted in place. Both counts are lower and upper bounds: the overflow is certain."""
    dims, v, n, R, vfov = (130, 130, 130), 0.1, 9, 60, 150.0
    rng = np.random.default_rng(7)
    pos = _tree(rng, n + 1, dims, v, 3.0)[1]
    parent = np.array([-1] + [0] * n, np.int32)  # one level of n nodes
    sensor = Sensor(100, vfov, 24, 16, R * v, yaws, 0.0)
    # bricks certainly inside the range and the elevation band of a node, for every group of 64 yaws
    c = np.stack(np.meshgrid(*[np.arange(0, d, 4) + 2.0 for d in dims], indexing="ij"), -1).reshape(-1, 3)
    records = 0
    for p in pos[1:] / v:
        d = c - p
        rho = np.hypot(d[:, 0], d[:, 1])
        far = np.sqrt((d ** 2).sum(1))
        inside = (far < R - 3.5) & (far > 12) & (np.abs(d[:, 2]) + 2 < math.tan(math.radians(vfov / 2)) * (rho - 3))
        records += int(inside.sum()) * (1 if mode == mig.MODE_PANORAMIC else -(-yaws // 64))
    share = {mig.MODE_INTERVAL: 0.7, mig.MODE_PANORAMIC: 0.5}.get(mode, 0.3)
    room = max(1 << 16, n * (int(share * (4.19 * ((R + 1) / 4 + 1.74) ** 3 + 1)) + 1))
    assert records > 1.05 * room
    m = mig.Map(ctx, np.zeros(dims[::-1], np.uint8), v)
    outs = []
    try:
        for kernel in (mig.COUNT_NODES, mig.COUNT_RAYS):
            ctx.set_count_kernel(kernel, 0)
            outs.append(mig.tree_eval(m, parent, pos, sensor, mode=mode, want_counts=True))
        for k in ("abs", "marg", "yaw", "cnt_abs", "cnt_marg"):
            assert np.array_equal(outs[0][k], outs[1][k]), k
        assert outs[0]["abs"].sum() > 0
    finally:
        ctx.set_count_kernel(mig.COUNT_AUTO, 0)
        m.close()
