"""The size rules of the pass kernels (csrc/plan.h) on the CPU: the radices of
lengths with a factor 3, and the tile every pass gets for a range of lengths,
row counts and precisions."""

import json
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"
LENGTHS = [24, 36, 48, 72, 96, 108, 144, 192, 288, 384, 576, 768, 1152, 1536, 2304, 3072, 64]


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("plan") / "plan_size_rules")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1707_09177_gb300", "csrc"), "-I" + CUDA_INC,
                    os.path.join(ROOT, "tests", "plan_size_rules.cpp"), "-o", exe], check=True)
    return json.loads(subprocess.run([exe] + [str(n) for n in LENGTHS], check=True, capture_output=True,
                                     text=True).stdout)


def test_fused_radices(rules):
    for n in LENGTHS:
        d = rules["fused"][str(n)]
        assert d["key64"] == 12                       # float64 keeps the separate radices
        if not d["ok"]:
            assert d["key"] == 12
            continue
        assert n % 3 == 0 and 36 <= n <= 2304 and d["key"] == 13
        r = d["r"]
        assert int(np.prod(r)) == n and len(r) <= 5 and all(12 % x == 0 for x in r) and d["rev"] == r[::-1]
        odd = [x % 3 == 0 for x in r]
        assert odd == sorted(odd)                     # powers of two first
    assert not rules["fused"]["24"]["ok"] and not rules["fused"]["3072"]["ok"] and not rules["fused"]["64"]["ok"]


def test_every_tile_is_one_the_kernels_run(rules):
    for L, nseq, cs, transposed, want, ok, E, W, T, ld, smem, stages in rules["tiles"]:
        if not ok:
            assert L in (8, 18), (L, nseq)            # rows too short for a block of whole butterflies
            continue
        assert W & (W - 1) == 0 and W * L == T * E and 1 <= T <= 256 and smem == W * ld * cs <= 112 * 1024
        assert E in (4, 12, 16, 24) and 1 <= stages <= 5
        last = L                                      # rows hold L + 1 elements
        assert ld > last + last // 16
        if transposed:
            assert nseq % W == 0
            B = 128 // cs
            if 1 < W < B:                             # a phase of W rows x B/W elements: distinct banks
                assert sorted((w * ld + k) % B for w in range(W) for k in range(B // W)) == list(range(B))
            else:
                assert W == 1 or ld % 2 == 1
        else:
            assert ld % 2 == 1
