"""The bounds-checked build checks what the default counts read and write: brick masks and distances, step
counts, tile and depth bounds, the queue of undecided bricks and the ancestors' depth buffers. Each kind in
turn is declared half as large as it is (MIG_BOUNDS_HALF, only read by that build), so that accesses to its
upper half, all inside the buffer, must be reported; with the true sizes nothing is."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import os, sys
import numpy as np
sys.path.insert(0, ROOT_DIR)
from paper_2609_40297_gb300 import _build
import paper_2609_40297_gb300 as mig
mig.LIB_PATH = _build.LIB_CHECKED
from synth import Sensor
assert mig.lib().mig_build_flags() == mig.BUILD_CHECKED
rng = np.random.default_rng(7)
dims, v, n = (130, 130, 130), 0.1, 9
pos = ((np.array(dims) / 2 + rng.uniform(-3, 3, (3 * n, 3))) * v).astype(np.float32)
parent = np.array([-1] + [0] * (n - 1) + list(range(1, n)) * 2 + [1, 2], np.int32)  # two levels of internal nodes
sensor = Sensor(100, 150, 24, 16, 6.0, 8, 0.0)
with mig.Context(0) as ctx:
    ctx.set_count_kernel(mig.COUNT_NODES, 0)
    m = mig.Map(ctx, np.zeros(dims[::-1], np.uint8), v)
    for mode in (mig.MODE_MARGINAL, mig.MODE_INTERVAL, mig.MODE_PANORAMIC):
        for kind in (0, 4, 8, 16, 32, 64, 0):
            os.environ["MIG_BOUNDS_HALF"] = str(kind)
            try:
                mig.tree_eval(m, parent, pos, sensor, mode=mode)
                said = 0
            except mig.MigError as e:
                assert e.status == mig.MIG_ECUDA and "bounds check" in str(e)
                said = int(str(e).split("kinds ")[1].split(")")[0])
            assert said == kind, (mode, kind, said)
    m.close()
print("kinds ok")
"""


def test_every_kind_of_buffer_is_checked():
    from paper_2609_40297_gb300 import _build
    _build.build(checked=True)
    r = subprocess.run([sys.executable, "-c", CHILD.replace("ROOT_DIR", repr(ROOT))], capture_output=True, text=True,
                       timeout=1200)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "kinds ok" in r.stdout
