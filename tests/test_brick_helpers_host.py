"""CPU tests of the brick steps (csrc/bricks.cuh), compiled for the host: the cast's jumps and exact
walk against a plain DDA, the whole-box camera verdicts against every voxel of the box in exact
integers, and the float visit decisions against the exact visit test. Each must never disagree: the
whole-brick verdicts, the certain visits and the slab test stand in for the exact tests."""
import os
import re
import subprocess

import pytest

from test_kernel_helpers_host import HERE, ROOT, _nvcc


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    out = str(tmp_path_factory.mktemp("bricks") / "brick_helpers_check")
    cmd = [nvcc, "-x", "cu", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2609_40297_gb300", "csrc"),
           "-I", os.path.join(ROOT, "include"), os.path.join(HERE, "brick_helpers_check.cu"), "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return out


@pytest.mark.parametrize("seed", [1, 2])
def test_brick_steps_agree_with_their_definitions(program, seed):
    r = subprocess.run([program, str(seed)], capture_output=True, text=True, timeout=600)
    c = {k: int(v) for k, v in re.findall(r"(\w+) (\d+)", r.stdout)}
    assert r.returncode == 0, r.stdout[-2000:]
    assert c["hits"] > 10_000 and c["inside"] > 10_000 and c["outside"] > 10_000 and c["sure"] > 1_000_000
    assert c["beam_free"] > 10_000 and c["beam_rays"] - c["beam_free"] > 100_000
    assert c["cast_bad"] == c["beam_bad"] == c["box_bad"] == c["sure_bad"] == c["slab_bad"] == 0
    assert c["undecided"] < 0.002 * c["slabs"]
