"""CPU test that no compile-time option selects another voxel layout than the x-fastest rows which the
brick masks and distances are made from and allocated behind: a build with another one would read and write
beyond the map's allocation."""
import os
import subprocess

import pytest

from test_kernel_helpers_host import ROOT, _nvcc

CSRC = os.path.join(ROOT, "paper_2609_40297_gb300", "csrc")


@pytest.mark.parametrize("source", ["kernels.cu", "nodecount.cu"])
def test_layout_is_not_an_option(source):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    out = [subprocess.run([nvcc, "-E", "-std=c++17", "-arch=compute_103a", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                           *extra, os.path.join(CSRC, source)], capture_output=True, text=True, check=True).stdout
           for extra in ([], ["-DMIG_LAYOUT=0"])]
    assert out[0] and out[0] == out[1]
