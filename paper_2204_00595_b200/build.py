"""Build libmonarch.so in-tree with nvcc for sm_100a (cross-compiles without a GPU)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB = os.path.join(_PKG, "libmonarch.so")
PYCALLS = os.path.join(_PKG, "_pycalls.so")      # argument marshalling of the hot calls (plain C, CPython API)

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC",
    "-cudart", "static",
    "--threads", "0",          # one compile job per source file
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _build_pycalls() -> None:
    src = os.path.join(CSRC, "pycalls.c")
    deps = [src, os.path.join(_ROOT, "include", "monarch.h"), os.path.abspath(__file__)]
    if os.path.exists(PYCALLS) and all(os.path.getmtime(d) <= os.path.getmtime(PYCALLS) for d in deps):
        return
    tmp = PYCALLS + f".tmp{os.getpid()}"
    subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"],
                    "-I", os.path.join(_ROOT, "include"), "-o", tmp, src], check=True)
    os.replace(tmp, PYCALLS)


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(
        os.path.join(_ROOT, "include", "*.h")) + [os.path.abspath(__file__)]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into libmonarch.so and pycalls.c into _pycalls.so (only if sources changed)."""
    _build_pycalls()
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc] + NVCC_FLAGS + ["-I", os.path.join(_ROOT, "include"), "-I", CSRC,
                                 "-shared", "-o", tmp] + sources()
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
        print(" ".join(cmd), file=sys.stderr)
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
