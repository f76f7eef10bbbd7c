"""The work counters of a launch of the fused engine (host logic, no GPU): the
library's own accumulator, compiled for the host, holds the longest launch that
a forest's budget allows."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <cstdio>
#include "dvc_pool.cuh"
int main() {
    dvc::WorkSum w{0ull, 0ull};
    for (int it = 0; it < (1 << 24); ++it) w.add(27u, 416u);  // a warp's pass over 32 two-player games
    dvc::WorkSum one{0xFFFFFFFFull, 0xFFFFFFFFull};
    one.add(1u, 2u);
    std::printf("%llu %llu %llu %llu\n", w.words, w.steps, one.words, one.steps);
    return 0;
}
'''


def test_longest_launch_does_not_wrap(tmp_path):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "w.cu", tmp_path / "w"
    src.write_text(SRC)
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                    "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_2403_10720_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(x) for x in out] == [27 << 24, 416 << 24, 1 << 32, (1 << 32) + 1]
