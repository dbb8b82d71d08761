"""Builds the CUDA library libgad.so in-tree for sm_103a with nvcc.

The translation units (host driver, pass kernels per precision and element count, the
multi-group pass kernels of batched solves, the allocation-free filter, the
learned guess's warp-level and tcgen05 kernels) compile in parallel; the result is linked into
paper_1707_09177_gb300/libgad.so next to this file.
"""

from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libgad.so")
# (source, defines): the pass kernels are one unit per precision and per-thread
# element count, the longest to compile first
SOURCES = ([("kernels_e.cu", ("GAD_REAL=float", "GAD_E=16")), ("kernels_multi.cu", ("GAD_E=16",))]
           + [("kernels_e.cu", ("GAD_REAL=%s" % t, "GAD_E=%d" % e)) for t in ("float", "double") for e in (24, 16, 12, 4)
              if (t, e) != ("float", 16)]
           + [("kernels_multi.cu", ("GAD_E=%d" % e,)) for e in (24, 12, 4)]
           + [("kernels_fused.cu", ("GAD_LONG=%d" % g,)) for g in (1, 0)]
           + [("kernels_cluster.cu", ("GAD_REAL=%s" % t,)) for t in ("float", "double")]
           + [(f, ()) for f in ("api.cu", "kernels_f32.cu", "kernels_f64.cu", "noalloc.cu", "cnn.cu", "conv_tc.cu")])
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc():
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found; the CUDA toolkit is required to build libgad.so")
    return cand


def _flags():
    return ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC",
                   "-I" + os.path.join(ROOT, "include")]


def _compile(src, verbose):
    src, defines = src
    name = "_".join([os.path.splitext(src)[0]] + [d.split("=")[1] for d in defines])
    obj = os.path.join(BUILD, name + ".o")
    cmd = [_nvcc()] + _flags() + ["-D" + d for d in defines] + ["-c", os.path.join(CSRC, src), "-o", obj]
    if verbose:
        cmd.insert(1, "-Xptxas=-v")
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, r.stdout, r.stderr))
    return obj, r.stderr


def build(verbose=False, force=False):
    """Compiles and links libgad.so; returns its path."""
    os.makedirs(BUILD, exist_ok=True)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "gad.h")]
    if (not force and os.path.exists(LIB)
            and os.path.getmtime(LIB) > max(os.path.getmtime(d) for d in deps)):
        return LIB
    with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 8)) as ex:
        results = list(ex.map(lambda s: _compile(s, verbose), SOURCES))
    if verbose:
        for _, log in results:
            sys.stderr.write(log)
    objs = [o for o, _ in results]
    tmp = LIB + ".tmp"
    cmd = [_nvcc()] + ARCH + ["-shared", "-o", tmp] + objs
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s\n%s" % (r.stdout, r.stderr))
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
