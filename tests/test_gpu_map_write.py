"""What a map update derives from the codes (masks and distances of the 4x4x4 bricks, occupancy bytes of the
8x8x8 bricks and super-bricks), seen through the counts that use it: after updates of one to a few voxels,
in grids of one brick, of odd sides and of more than one word of bricks along x, the per-node count and the
persistent batch kernel on the updated map equal the ray-by-ray count on a map made afresh."""
import numpy as np
import pytest

import synth
from synth import Sensor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2609_40297_gb300 as mig  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = mig.Context(0, stream=torch.cuda.Stream())
    yield c
    c.close()


@pytest.mark.parametrize("dims", [(3, 4, 2), (33, 29, 17), (131, 34, 36), (290, 20, 9), (64, 64, 32)])
def test_small_updates(ctx, dims):
    nx, ny, nz = dims
    rng = np.random.default_rng(nx)
    v, n = 0.1, 10
    grid = np.where(rng.random((nz, ny, nx)) < 0.6, 0, 1).astype(np.uint8)
    m = mig.Map(ctx, grid, v)
    pos = (rng.uniform(0.05, 0.95, (n, 3)) * np.array(dims) * v).astype(np.float32)
    parent = np.array([-1] + [int(rng.integers(0, i)) for i in range(1, n)], np.int32)
    sensor = Sensor(90, 60, 40, 30, min(0.1 * max(dims), 9.0), 6, 0.0)
    tiles = ctx.get_tiles()
    try:
        spots = [(int(rng.integers(0, nx)), int(rng.integers(0, ny)), int(rng.integers(0, nz))) for _ in range(10)]
        spots[:4] = [(nx - 1, ny - 1, nz - 1), (0, 0, 0), (min(31, nx - 1), 0, 0), (min(128, nx - 1), ny - 1, 0)]
        for i in range(2 * len(spots)):  # every spot is occupied, later freed
            x, y, z = spots[i % len(spots)]
            d = [int(rng.integers(1, 4)) for _ in range(3)]
            d = [min(e, s - o) for e, s, o in zip(d, dims, (x, y, z))]
            box = np.full(d[::-1], 2 if i < len(spots) else int(rng.integers(0, 2)), np.uint8)
            m.update(x, y, z, box)
            grid[z:z + d[2], y:y + d[1], x:x + d[0]] = box
            if i % 3 and i != 2 * len(spots) - 1:
                continue
            fresh = mig.Map(ctx, grid, v)
            try:
                ctx.set_count_kernel(mig.COUNT_RAYS, 0)
                ref = mig.tree_eval(fresh, parent, pos, sensor, want_counts=True, want_depth=True)
                ctx.set_count_kernel(mig.COUNT_NODES, 0)
                got = mig.tree_eval(m, parent, pos, sensor, want_counts=True, want_depth=True)
                for k in ("abs", "marg", "yaw", "cnt_abs", "cnt_marg", "depth"):
                    assert np.array_equal(got[k], ref[k]), (i, k)
                ctx.set_count_kernel(mig.COUNT_AUTO, 0)
                ctx.set_tiles(tiles[0], tiles[1], tiles[2], 0)
                for got in mig.tree_eval_batch(ctx, [(parent, pos, sensor)] * 2, [m, m]):
                    for k in ("abs", "marg", "yaw"):
                        assert np.array_equal(got[k], ref[k]), (i, k)
            finally:
                ctx.set_count_kernel(mig.COUNT_AUTO, 0)
                ctx.set_tiles(*tiles)
                fresh.close()
        assert np.array_equal(m.read(), grid)
    finally:
        m.close()
