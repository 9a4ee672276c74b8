"""Nodes in clutter, where rays are cast voxel by voxel up to the first free brick: the counts and depth
buffers equal those of the ray-by-ray count, whose depth buffers are cast one ray at a time as well, on maps
with occupied voxels in nearly every brick, free corridors through them, odd sides and nodes at the grid's
edges, in every mode; and the oracle's."""
import numpy as np
import pytest

import oracle
from synth import Sensor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2609_40297_gb300 as mig  # noqa: E402

MODES = (mig.MODE_MARGINAL, mig.MODE_ABSOLUTE, mig.MODE_INTERVAL, mig.MODE_PANORAMIC)


@pytest.fixture(scope="module")
def ctx():
    c = mig.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("dims,share,image", [
    ((41, 38, 21), 0.03, (33, 21)), ((41, 38, 21), 0.3, (130, 70)), ((18, 22, 10), 0.05, (48, 36)), ((90, 70, 33), 0.04, (64, 40))])
def test_clutter(ctx, dims, share, image):
    nx, ny, nz = dims
    rng = np.random.default_rng(nx + int(100 * share))
    v, n = 0.2, 24
    grid = np.where(rng.random((nz, ny, nx)) < 0.5, 0, 1).astype(np.uint8)
    grid[rng.random((nz, ny, nx)) < share] = 2
    grid[nz // 2:nz // 2 + 6, :, nx // 3:nx // 3 + 6] = 1  # a free corridor
    pos = rng.uniform(0.0, 1.0, (n, 3)) * (np.array(dims) - 0.01)
    pos[::3] = np.floor(pos[::3])  # on voxel corners
    pos[:3] = [[0, 0, 0], [nx - 0.01, ny - 0.01, nz - 0.01], [nx / 2, 0, nz - 0.5]]
    pos = (pos * v).astype(np.float32)
    parent = np.array([-1] + [(i - 1) // 2 for i in range(1, n)], np.int32)
    sensor = Sensor(100, 80, image[0], image[1], 4.0, 5, 0.0)
    m = mig.Map(ctx, grid, v)
    try:
        for mode in MODES:
            outs = []
            for kernel in (mig.COUNT_NODES, mig.COUNT_RAYS):
                ctx.set_count_kernel(kernel, 0)
                outs.append(mig.tree_eval(m, parent, pos, sensor, mode=mode, want_counts=True, want_depth=True))
            for k in ("abs", "marg", "yaw", "cnt_abs", "cnt_marg", "depth"):
                assert np.array_equal(outs[0][k], outs[1][k]), (mode, k)
            ref = oracle.eval_tree(grid, v, (0, 0, 0), parent, pos, sensor, mode=mode, want_counts=True, want_depth=True)
            for k in ("abs", "marg", "yaw", "cnt_abs", "cnt_marg", "depth"):
                assert np.array_equal(outs[0][k], ref[k]), (mode, k)
            assert outs[0]["abs"].sum() > 0
    finally:
        ctx.set_count_kernel(mig.COUNT_AUTO, 0)
        m.close()


def test_bad_codes_are_refused(ctx):
    """Codes above 2 are refused wherever they stand, by create and update, and leave the map as it was."""
    grid = np.zeros((5, 7, 300), np.uint8)
    for at in (0, 127, 128, 5 * 7 * 300 - 1):
        bad = grid.copy()
        bad.reshape(-1)[at] = 3
        with pytest.raises(mig.MigError) as e:
            mig.Map(ctx, bad, 0.1)
        assert e.value.status == mig.MIG_EINVAL and f"index {at} " in str(e.value)
    m = mig.Map(ctx, grid, 0.1)
    try:
        box = np.full((2, 2, 200), 2, np.uint8)
        box.reshape(-1)[777] = 255
        with pytest.raises(mig.MigError) as e:
            m.update(0, 0, 0, box)
        assert e.value.status == mig.MIG_EINVAL and "index 777 " in str(e.value)
        assert np.array_equal(m.read(), grid)
    finally:
        m.close()
