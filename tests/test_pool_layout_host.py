"""Shared memory of the fused engine's CTAs (host logic, no GPU): the library's own
layout, compiled for the host, gives the word rings to the uniform playouts
only, and every shape that dvc_forest_tune takes fits."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r'''
#include <cstdio>
#include "dvc_pool.cuh"
int main() {
    for (int T = 1; T <= 64; ++T)
        for (int W = 1; W <= 32; ++W) {
            const dvc::PoolLayout u(T, W, false), o(T, W, true);
            std::printf("%d %u %u %u\n", W, u.bytes, o.bytes, o.ring);
        }
    return 0;
}
'''


def test_layout(tmp_path):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "l.cu", tmp_path / "l"
    src.write_text(SRC)
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                    "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_2403_10720_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    for line in out.splitlines():
        W, uniform, ordered, ring = map(int, line.split())
        assert ring == ordered                     # nothing behind where the rings would stand
        assert uniform - ordered == 19 * 128 * W   # 16 rows of words and three repeated
        assert uniform <= 200 * 1024
