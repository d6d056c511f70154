"""Host rules of the launch sequences, compiled and run on the CPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include <cstdio>
#include "rykov_launch.cuh"
int main() {
    // colour offsets of equal colours, and of one large colour among small ones
    std::vector<int> even{0, 256, 512}, large{0, 30000}, big{0, 40000, 80000};
    for (int c = 0; c < 15; ++c) large.push_back(large.back() + 1);
    for (int ms : {4, 6})
        for (const auto* c : {&even, &large, &big})
            std::printf("%d%d ", (int)rk::macro_ahead(*c, ms, true), (int)rk::macro_ahead(*c, ms, false));
    return 0;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_macro_phases_ahead_of_their_turn_by_the_largest_colour(tmp_path):
    src, exe = tmp_path / "rules.cu", tmp_path / "rules"
    src.write_text(PROGRAM)
    subprocess.run([NVCC, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2303_10846_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["11", "01", "01"] * 2
