"""The digests that tie the committed profiles to the kernels cover every file of the library that a
kernel's file includes, directly or not (as the compiler sees them)."""
import os
import subprocess

import pytest

import bench
from paper_1411_6697_gb300 import build


@pytest.mark.parametrize("kernel", sorted(bench.PROFILE))
def test_every_included_file_counts(kernel):
    csrc = os.path.join(os.path.dirname(os.path.abspath(build.__file__)), "csrc")
    root = {"march": "march.cu", "step": "tile.cu", "batch": "batch.cu"}[kernel]
    made = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-MM", os.path.join(csrc, root)], check=True,
                          capture_output=True, text=True).stdout
    files = {os.path.basename(f) for f in made.replace("\\", " ").split() if os.path.dirname(os.path.abspath(f)) == csrc}
    assert files == set(bench.step_kernel_sources(kernel))
