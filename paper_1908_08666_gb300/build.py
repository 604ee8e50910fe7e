"""Build libhhgs.so in-tree with nvcc for sm_103a (translation units compiled in parallel)."""

from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "_build")
LIB = os.path.join(OUT, "libhhgs.so")

# many instantiations of unrolled kernels: ptxas in parallel.  Not for the other files: parallel ptxas made
# the mma.sync convolution slower (forward pass on 33^3 voxels 65 -> 71 us).
SPLIT = ["hhg_sweep_f32.cu", "hhg_sweep_f64.cu", "hhg_stokes_f32.cu", "hhg_stokes_f64.cu", "hhg_rows_f32.cu",
         "hhg_rows_f64.cu"]
SOURCES = ["hhg_host.cpp", "hhg_solve.cpp", "hhg_learn.cpp", "hhg_sweep.cu", "hhg_gs.cu", "hhg_vec.cu", "hhg_learn.cu",
           "hhg_twod.cu", *SPLIT]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC,-O2",
         "-I" + os.path.join(os.path.dirname(HERE), "include")]


def nvcc():
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found")
    return exe


def _compile(src, extra):
    obj = os.path.join(OUT, src + ".o")
    split = ["--split-compile", "0"] if src in SPLIT else []
    cmd = [nvcc(), *ARCH, *FLAGS, *split, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed for %s:\n%s\n%s" % (src, " ".join(cmd), r.stderr))
    return obj, r.stderr


def build(verbose=False, extra=()):
    os.makedirs(OUT, exist_ok=True)
    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        res = list(ex.map(lambda s: _compile(s, list(extra)), SOURCES))
    objs = [o for o, _ in res]
    if verbose:
        for _, err in res:
            if err:
                sys.stderr.write(err)
    tmp = LIB + ".tmp"
    cmd = [nvcc(), *ARCH, "-shared", "-cudart", "static", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n%s" % r.stderr)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    extra = sys.argv[1:]
    print(build(verbose=True, extra=extra))
