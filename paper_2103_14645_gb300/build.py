"""Build the in-tree renderer library libsnerg.so for sm_103a with nvcc.

Each translation unit compiles in parallel into _build/ (the kernels of the march once per
block build), then nvcc links the shared
library next to this file. Only the sm_103a target is emitted (one -gencode).
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(HERE, "libsnerg.so")
SOURCES = ["snerg_api.cu", "snerg_prep.cu", "snerg_noalloc.cu", "snerg_train.cu", "snerg_bake.cu"]
# compiled once per block build: log2 of the block edge as a constant (0: any edge), and whether
# channel 0 holds alpha (2: by the scene's flags)
PER_BLOCK_SOURCES = ["snerg_fwd.cu", "snerg_bwd.cu"]
BLOCK_BUILDS = [(0, 2)] + [(lgb, alpha) for lgb in (3, 4, 5, 6) for alpha in (0, 1)]
UNITS = [(f, b) for f in PER_BLOCK_SOURCES for b in BLOCK_BUILDS] + [(f, None) for f in SOURCES]
GENCODE = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for p in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc"):
        if p and os.path.exists(p):
            return p
    return "nvcc"


def _flags(extra=()):
    return [*GENCODE, "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-O2",
            "-I", INCLUDE, "-I", CSRC, *extra]


def _compile(unit, extra, verbose: bool) -> str:
    src, block = unit
    obj = os.path.join(BUILD, os.path.splitext(src)[0] + ("" if block is None else "_%d_%d" % block) + ".o")
    define = [] if block is None else ["-DSNERG_LGB=%d" % block[0], "-DSNERG_ALPHA=%d" % block[1]]
    cmd = [nvcc(), *_flags(extra), *define, "-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
    if r.returncode:
        raise RuntimeError(f"nvcc failed on {src}")
    return obj


def build(verbose: bool = False, extra=()) -> str:
    os.makedirs(BUILD, exist_ok=True)
    with cf.ThreadPoolExecutor(max_workers=os.cpu_count() or 4) as ex:
        objs = list(ex.map(lambda u: _compile(u, extra, verbose), UNITS))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc(), *GENCODE, "-shared", "-cudart", "static", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode:
        sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
    if r.returncode:
        raise RuntimeError("nvcc link failed")
    os.replace(tmp, LIB)
    return LIB


def sources_newer_than_lib() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "snerg.h")]
    return any(os.path.getmtime(f) > t for f in files)


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, extra=["-Xptxas", "-v"] if "--ptxas" in sys.argv else []))
