"""Which snapshots the packing kernel may take: only memory of the handle's own device, with that device
current. Compiled from the library's header for the host, so devices that this machine does not have can
be named."""
import os
import subprocess

from paper_1411_6697_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.abspath(build.__file__)), "csrc")
PROGRAM = r"""
#include "kernels.cuh"
#include <cstdio>
int main()
{
    // dst device, state device, current device
    const int d[5][3] = {{0, 0, 0}, {1, 0, 1}, {0, 0, 1}, {1, 0, 0}, {1, 1, 1}};
    for (const auto& r : d) std::printf("%d", (int)lbk::pack_there(8, 4096, true, r[0], r[1], r[2]));
    std::printf(" %d %d\n", (int)lbk::pack_there(8, 4100, true, 0, 0, 0), (int)lbk::pack_there(8, 4096, false, 0, 0, 0));
}
"""


def test_only_on_the_state_s_device(tmp_path):
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True, capture_output=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["10001", "0", "0"]
