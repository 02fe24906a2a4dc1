"""Builds libbsp.so (the C-ABI CUDA library, nvcc for sm_100a) and _bsp_native.so (the binding's argument
marshalling, against the installed torch) in-tree."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
INCLUDE = os.path.join(os.path.dirname(PKG_DIR), "include")
LIB_PATH = os.path.join(PKG_DIR, "libbsp.so")
NATIVE_SRC = os.path.join(CSRC, "bsp_native.cpp")
NATIVE_PATH = os.path.join(PKG_DIR, "_bsp_native.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo", "--threads", "0",
    "-Xcompiler", "-fPIC", "-shared",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(NATIVE_PATH):
        return True
    built = min(os.path.getmtime(LIB_PATH), os.path.getmtime(NATIVE_PATH))
    deps = sources() + [NATIVE_SRC] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(p) > built for p in deps)


def _run(cmd, verbose: bool, what: str) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"compiling {what} failed")


def build_native(verbose: bool = False) -> str:
    """Compile the binding's marshalling module against libbsp.so and the installed torch."""
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = [shutil.which("g++") or "g++", "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-isystem", os.path.join(root, "include"), "-isystem", os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-isystem", os.path.join(cuda, "include"), "-isystem", sysconfig.get_paths()["include"], "-I", INCLUDE,
           NATIVE_SRC, "-o", NATIVE_PATH + ".tmp", "-L", PKG_DIR, "-l:libbsp.so", "-Wl,-rpath,$ORIGIN",
           "-L", os.path.join(root, "lib"), "-lc10", "-lc10_cuda", "-ltorch_python"]
    _run(cmd, verbose, "_bsp_native.so")
    os.replace(NATIVE_PATH + ".tmp", NATIVE_PATH)
    return NATIVE_PATH


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into libbsp.so, then the marshalling module; returns the library path."""
    if not force and not is_stale():
        return LIB_PATH
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        raise RuntimeError("nvcc not found: cannot build libbsp.so")
    cmd = [nvcc, *NVCC_FLAGS, "-I", INCLUDE, "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += ["-o", LIB_PATH + ".tmp", *sources()]
    _run(cmd, verbose, "libbsp.so")
    os.replace(LIB_PATH + ".tmp", LIB_PATH)
    build_native(verbose)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
