"""Compile the CUDA library for sm_100a into paper_2202_07471_b200/libsquant.so (in-tree)."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsquant.so")
LIB_DEBUG = os.path.join(HERE, "libsquant_debug.so")   # the checked build (-DSQUANT_DEBUG_BOUNDS), for tests on small cases
SOURCES = [os.path.join(CSRC, "squant.cu")]
DEPS = SOURCES + sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + [os.path.join(ROOT, "include", "squant.h")]

# -fmad=false: the solver's fp32 steps (division, rounding, difference) are written with
# explicit round-to-nearest intrinsics; no contraction is wanted anywhere else either.
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
              "-fmad=false", "--shared", "-Xcompiler", "-fPIC", "-Xptxas", "-v",
              "-I", os.path.join(ROOT, "include"), "-I", CSRC]


def nvcc_path() -> str:
    p = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(p):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    return p


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    lib = LIB_DEBUG if debug else LIB
    if not force and os.path.exists(lib) and all(
            os.path.getmtime(lib) >= os.path.getmtime(d) for d in DEPS):
        return lib
    tmp = lib + f".tmp{os.getpid()}"
    cmd = [nvcc_path(), *NVCC_FLAGS, *(["-DSQUANT_DEBUG_BOUNDS"] if debug else []), "-o", tmp, *SOURCES]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        print(res.stdout)
        print(res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building " + os.path.basename(lib))
    os.replace(tmp, lib)
    return lib


MARSHAL = os.path.join(HERE, "_marshal.so")            # Python extension: descriptors of LayerBuffers objects
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")


def build_marshal(force: bool = False) -> str:
    if not force and os.path.exists(MARSHAL) and all(
            os.path.getmtime(MARSHAL) >= os.path.getmtime(d) for d in (MARSHAL_SRC, os.path.join(ROOT, "include", "squant.h"))):
        return MARSHAL
    import sysconfig
    import torch
    base = os.path.dirname(torch.__file__)
    tmp = MARSHAL + f".tmp{os.getpid()}"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"],
           "-isystem", os.path.join(base, "include"), "-isystem", os.path.join(base, "include", "torch", "csrc", "api", "include"),
           "-o", tmp, MARSHAL_SRC, "-L", os.path.join(base, "lib"), "-lc10", "-ltorch_cpu", "-ltorch_python"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        print(res.stdout)
        print(res.stderr)
        raise RuntimeError("g++ failed building _marshal.so")
    os.replace(tmp, MARSHAL)
    return MARSHAL


if __name__ == "__main__":
    print(build(force=True, verbose=True))
    print(build_marshal(force=True))
    print(build(force=True, debug=True))
