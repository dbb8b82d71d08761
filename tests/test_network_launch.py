"""The launch rule of the network's output layer (csrc/cnn.h) on the CPU: small
grids spread over the SMs instead of marching through eight planes on a few."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"
SRC = """
#include <cstdio>
#include "cnn.h"
int main() {
  for (int Z : {3, 8, 18, 24, 64, 256, 512})
    for (long long columns : {1LL, 3LL, 30LL, 151LL, 152LL, 1000LL, 100000LL})
      std::printf("%d %lld %d\\n", Z, columns, gad::out_planes(columns, Z));
}
"""


def test_small_grids_use_the_gpu(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run([gxx, "-std=c++17", "-I" + os.path.join(ROOT, "paper_1707_09177_gb300", "csrc"), "-I" + CUDA_INC,
                    str(tmp_path / "t.cpp"), "-o", exe], check=True)
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        Z, columns, zc = map(int, line.split())
        blocks = columns * -(-Z // zc)
        assert 1 <= zc <= Z
        assert blocks >= 152 or zc == 1, line        # a block per SM, or nothing left to split
        if zc < 5 and zc < Z:                         # halving from above 8 ends at 5 to 8; shorter only where needed
            assert columns * -(-Z // (2 * zc)) < 152, line
