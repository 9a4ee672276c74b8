"""CPU test of how the device code reads what it has written. The kernels of a level are launched before
the ones ahead of them have ended (csrc/launch.cuh), and the persistent kernel's CTAs read one another's
results, so the read-only path (__ldg) is allowed for the map and the camera tables only: step counts, tile
bounds and depth buffers take ordinary loads. Read from the sources: run on a GPU, a stale value shows by
chance only."""
import glob
import os
import re

from test_kernel_helpers_host import ROOT

CSRC = os.path.join(ROOT, "paper_2609_40297_gb300", "csrc")
# voxel codes, map masks and distances (through ld_u8 and ld_u64), rows of the yaw table
READ_ONLY = {"dev_path.cuh": {"g + a", "row", "row + 1", "row + 2"}, "voxitems.cuh": {"row", "row + 1", "row + 2"},
             "voxcount.cuh": {"p"}, "bricks.cuh": {"reinterpret_cast<const unsigned long long *>(p)"}}


def _calls(text, name):
    """The arguments of the calls of `name` (balanced parentheses)."""
    for m in re.finditer(rf"\b{name}\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]


def test_read_only_loads_are_of_the_map_and_the_camera():
    found = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        args = set(_calls(text, "__ldg"))
        if args:
            found[os.path.basename(path)] = args
        for name in ("ld_u8", "ld_u64"):  # a parameter in their own definition
            for a in _calls(text, name):
                assert not re.search(r"steps|hz|pyr|depths|arena|\bD\b", a), (path, name, a)
    assert found == READ_ONLY
