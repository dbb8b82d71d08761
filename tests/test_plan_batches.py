"""How the tiles of a grid's passes follow the batch (csrc/plan.h), on the CPU:
what fixes a field's result never does, and the launches without dots take
the wide tiles again once the batch alone fills the GPU."""

import json
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"
SIDES = [8, 12, 24, 32, 48, 64, 72, 96, 128, 144, 192, 256, 288, 512, 768, 1024, 2048, 2304, 4096]


def _grids():
    g = [(nx, ny, 1) for nx in SIDES for ny in SIDES + [18, 54] if max(nx, ny) <= 16 * min(nx, ny)]
    three = [8, 24, 32, 48, 64, 72, 96, 128]
    return g + [(nx, ny, nz) for nx in three for ny in three for nz in three + [18]]


@pytest.fixture(scope="module")
def tiles(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("plan") / "plan_batch_rules")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1707_09177_gb300", "csrc"), "-I" + CUDA_INC,
                    os.path.join(ROOT, "tests", "plan_batch_rules.cpp"), "-o", exe], check=True)
    out = {}
    for cs in (8, 16):
        args = ["%d,%d,%d,%d" % (g + (cs,)) for g in _grids()]
        for r in json.loads(subprocess.run([exe] + args, check=True, capture_output=True, text=True).stdout):
            out[tuple(r["grid"]), r["cs"], r["batch"]] = r
    return out


def test_the_batch_changes_no_result(tiles):
    """Element counts (radices) and the tiles of launches with dots are the same
    in every batch; with and without dots a pass has one element count."""
    for (grid, cs, batch), r in tiles.items():
        one = tiles[grid, cs, 1]
        assert r["ok"] == one["ok"], (grid, cs)
        if not r["ok"]:
            continue
        for k in ("xi", "fl"):
            assert r[k] == one[k], (grid, cs, batch, k)
            assert r[k + "_nodots"][0] == r[k][0], (grid, cs, batch, k)
        for k in ("xf", "y"):
            assert r[k][0] == one[k][0], (grid, cs, batch, k)


def test_a_full_launch_has_no_narrow_tiles(tiles):
    """1024 fields fill the GPU with any tile: no pass without dots is narrower
    than half the block size it would take on a large grid (half, because widths
    are powers of two), unless a row of the next width would not fit."""
    want = {"xf": lambda nx: 128 if nx % 3 == 0 else 64, "xi_nodots": lambda nx: 256, "fl_nodots": lambda nx: 128,
            "y": lambda nx: 256}
    for (grid, cs, batch), r in tiles.items():
        if batch != 1024 or not r["ok"]:
            continue
        nx, ny, nz = grid
        for k, w in want.items():
            if k == "y" and nz == 1:
                continue
            E, W, T, ld, smem = r[k]
            L = {"xf": nx // 2, "xi_nodots": nx // 2, "y": ny}.get(k, nz if nz > 1 else ny)
            rows = {"xf": ny, "xi_nodots": ny, "y": nz}.get(k)
            if 2 * T > w(nx // 2) or 2 * smem > 100 * 1024:
                continue
            assert rows is not None and rows % (2 * W) != 0, (grid, cs, k, r[k])
    # the filter pass of a batch of 96 x 72 x 72 float64 fields
    assert tiles[(96, 72, 72), 16, 16]["fl_nodots"][2] >= 96
    assert tiles[(96, 72, 72), 16, 1]["fl"][2] < 96


def test_few_elements_per_thread_only_where_a_batch_gains_too(tiles):
    """4 elements per thread (radices 4 and 2) in float64 on small grids only:
    batches of float32 fields and of larger float64 ones are slower with them."""
    for (grid, cs, batch), r in tiles.items():
        if not r["ok"]:
            continue
        for k, kx in (("xf", grid[0] // 2), ("xi", grid[0] // 2), ("fl", grid[0] // 2 + 1), ("y", grid[0] // 2 + 1)):
            if r[k][0] == 4:
                assert cs == 16 and kx * grid[1] * grid[2] < 152 * 16 * 16, (grid, cs, k)
    assert tiles[(512, 512, 1), 8, 16]["fl"][0] == tiles[(64, 64, 64), 8, 1]["fl"][0] == 16
    assert tiles[(256, 256, 1), 16, 1]["fl"][0] == 4 and tiles[(64, 64, 64), 16, 1]["fl"][0] == 16


def test_blocks_wanted_of_a_launch_without_dots(tiles):
    """A launch keeps a wide tile only where that gives two blocks per SM, four
    for float64 powers of two."""
    for (grid, cs, batch), r in tiles.items():
        nx, ny, nz = grid
        if not r["ok"]:
            continue
        L, seqs = (nz, (nx // 2 + 1) * ny) if nz > 1 else (ny, nx // 2 + 1)
        E, W, T = r["fl_nodots"][:3]
        want = 152 * (4 if cs == 16 and L % 3 else 2)
        assert -(-seqs // W) * batch >= want or W == 1 or T // 2 < 32, (grid, cs, batch, r["fl_nodots"])
    assert tiles[(64, 64, 64), 16, 3]["fl_nodots"][1] < tiles[(64, 64, 64), 16, 16]["fl_nodots"][1]
