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
MARSHAL = os.path.join(HERE, "rmm_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))  # another interpreter builds its own
MARSHAL_SRC = os.path.join(CSRC, "marshal.c")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-Wall", "--expt-relaxed-constexpr",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target: str, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _headers():
    return glob.glob(os.path.join(ROOT, "include", "*.h"))


def stale() -> bool:
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers())


def marshal_stale() -> bool:
    return _older(MARSHAL, [MARSHAL_SRC] + _headers())


def build(force: bool = False, verbose: bool = False) -> str:
    if force or stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        extra = os.environ.get("RMM_NVCC_EXTRA", "").split()  # e.g. -DRMM_GEMM_STAMPS for the debug time stamps
        cmd = [nvcc, *NVCC_FLAGS, *extra, "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", LIB, *sources(),
               "-lcudart"]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
            print(" ".join(cmd), file=sys.stderr)
        subprocess.run(cmd, check=True)
    if force or marshal_stale():
        build_marshal()
    return LIB


def build_marshal() -> str:
    subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                    "-I", os.path.join(ROOT, "include"), "-o", MARSHAL, MARSHAL_SRC], check=True)
    return MARSHAL


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
