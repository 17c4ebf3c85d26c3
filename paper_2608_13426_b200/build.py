"""Build librmm_b200.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the binding's marshalling module."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "librmm_b200.so")
MARSHAL = os.path.join(HERE, "rmm_marshal.so")
MARSHAL_SRC = os.path.join(CSRC, "marshal.c")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "--expt-relaxed-constexpr",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(MARSHAL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(MARSHAL))
    deps = [MARSHAL_SRC] + sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    extra = os.environ.get("RMM_NVCC_EXTRA", "").split()  # e.g. -DRMM_GEMM_STAMPS for the debug time stamps
    cmd = [nvcc, *NVCC_FLAGS, *extra, "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", LIB, *sources(),
           "-lcudart"]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
        print(" ".join(cmd), file=sys.stderr)
    subprocess.run(cmd, check=True)
    build_marshal()
    return LIB


def build_marshal() -> str:
    subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                    "-I", os.path.join(ROOT, "include"), "-o", MARSHAL, MARSHAL_SRC], check=True)
    return MARSHAL


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
