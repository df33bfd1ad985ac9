"""The strip height of the FP32 2-D step, chosen anew at every launch: the heights tried give the choice of
a scan over all of them and stay few on tall grids. The rule is compiled from the library's header."""
import os
import subprocess

from paper_1411_6697_gb300 import build

CSRC = os.path.join(os.path.dirname(os.path.abspath(build.__file__)), "csrc")
PROGRAM = r"""
#include "kernels.cuh"
#include <cmath>
#include <cstdio>
int main()
{
    int differ = 0, many = 0;
    for (int G : {1, 7, 304})
        for (int nsx : {1, 3, 32})
            for (int ny : {1, 2, 3, 17, 64, 65, 517, 4096, 9999, 100003, 1000000}) {
                const int even = (ny + 1) & ~1;
                for (int cap : {even, even > 64 ? 64 : even}) {
                    auto cost = [&](long s, int r) {
                        const long rounds = (s + G - 1) / G;
                        return rounds * (r / 2 + 1.3) * (2 * s <= G ? 0.65 : 1.0) + 0.15 * (r / 2);
                    };
                    int tried = 0, rows = 2;
                    double best = 1e300;
                    for (int r = 2; r <= cap; r += 2) {
                        const double t = cost((long)nsx * ((ny + r - 1) / r), r);
                        if (t <= best) best = t, rows = r;
                    }
                    differ += lbk::march_rows(ny, cap, nsx, cost, &tried) != rows;
                    many += tried > 2 * std::sqrt((double)ny) + 3;
                }
            }
    std::printf("%d %d\n", differ, many);
}
"""


def test_few_heights_and_the_same_choice(tmp_path):
    src, exe = tmp_path / "plan.cu", tmp_path / "plan"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True,
                   capture_output=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0", "0"]
