"""A server's requests under a change of the count kernel: each keeps the kernel of its submission for its
device region and for its launches, so a request that is admitted after the change still returns what a
lone evaluation returns."""
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


@pytest.mark.parametrize("first,then", [(mig.COUNT_AUTO, mig.COUNT_PAIRS), (mig.COUNT_NODES, mig.COUNT_PAIRS),
                                        (mig.COUNT_PAIRS, mig.COUNT_NODES), (mig.COUNT_NODES, mig.COUNT_RAYS)])
def test_requests_keep_the_kernel_of_their_submission(first, then):
    """A long call holds the context; the change waits for it, then the server's worker does, woken by
    requests submitted before the change. Lock waiters are served in order, so the requests are admitted
    after it."""
    ctx = mig.Context(0, stream=torch.cuda.Stream())
    p = synth.random_small(131, nx=60, ny=60, nz=30, v=0.1, p_occ=0.001, n_nodes=24, max_depth=6,
                           sensor=Sensor(90, 60, 40, 30, 2.0, 8, 0.0))
    busy = synth.random_small(132, nx=60, ny=60, nz=30, v=0.1, p_occ=0.001, n_nodes=600, max_depth=12,
                              sensor=Sensor(90, 60, 320, 240, 2.0, 36, 0.0))
    m = mig.Map(ctx, p.map.grid, p.map.voxel_size, p.map.origin)
    modes = [mig.MODE_MARGINAL, mig.MODE_INTERVAL, mig.MODE_PANORAMIC, mig.MODE_SINGLE_PARENT]
    srv = mig.Server(ctx, arena_budget_bytes=1 << 30, max_inflight=4)
    try:
        want = [mig.tree_eval(m, p.tree.parent, p.tree.pos, p.sensor, mode=md) for md in modes]
        assert all(w["abs"].sum() > w["marg"].sum() > 0 for w in want)
        ctx.set_count_kernel(first, 0)
        holds = threading.Thread(target=mig.tree_eval_stats, args=(m, busy.tree.parent, busy.tree.pos, busy.sensor))
        change = threading.Thread(target=ctx.set_count_kernel, args=(then, 0))
        holds.start()
        time.sleep(0.02)
        change.start()
        time.sleep(0.02)
        subs = [srv.submit(m, p.tree.parent, p.tree.pos, p.sensor, mode=md) for md in modes]
        assert holds.is_alive() and change.is_alive()  # submitted before the change
        for t, _ in subs:
            assert srv.poll(t, timeout_us=30_000_000)
        holds.join()
        change.join()
        for (_, got), ref, md in zip(subs, want, modes):
            for k in ("abs", "marg", "yaw"):
                assert np.array_equal(got[k], ref[k]), (md, k)
    finally:
        srv.close()
        m.close()
        ctx.close()
