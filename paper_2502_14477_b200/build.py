"""Builds the C-ABI CUDA library in-tree with nvcc for sm_100a, and the native half of the Python binding
(a small extension module linked against it and against the installed torch) with g++."""
from __future__ import annotations

import glob
import os
import re
import shutil
import subprocess
import sys
import sysconfig

import torch

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libesa_b200.so")
NATIVE_SRC = os.path.join(CSRC, "esa_native.cpp")
INCLUDE_DIR = os.path.join(os.path.dirname(PKG_DIR), "include")


def native_path(python: str = sys.implementation.cache_tag, torch_version: str = torch.__version__) -> str:
    """File of the native module.  It is compiled against one torch and one Python, whose internals it reads, so both are
    part of its name: a module built against others is not found (and rebuilt), never loaded."""
    return os.path.join(PKG_DIR, "_esa_native.%s-torch%s.so" % (python, re.sub(r"[^0-9A-Za-z.]+", "_", torch_version)))


NATIVE_PATH = native_path()


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the ESA library is CUDA-only and cannot be built")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(INCLUDE_DIR, "*.h"))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(f) > t for f in deps)


def is_stale() -> bool:
    return _stale(LIB_PATH, _deps()) or _stale(NATIVE_PATH, [NATIVE_SRC, LIB_PATH])


def _run(cmd) -> str:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{os.path.basename(cmd[0])} failed:\n" + res.stdout + res.stderr)
    return res.stderr


def _build_native() -> None:
    tdir = os.path.dirname(torch.__file__)
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    _run([
        os.environ.get("CXX") or "g++", "-shared", "-fPIC", "-std=c++17", "-O2",
        f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
        "-I", sysconfig.get_paths()["include"], "-I", os.path.join(tdir, "include"),
        "-I", os.path.join(tdir, "include", "torch", "csrc", "api", "include"), "-I", cuda_inc,
        "-o", NATIVE_PATH, NATIVE_SRC,
        "-L", os.path.join(tdir, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python",
        "-L", PKG_DIR, "-l:" + os.path.basename(LIB_PATH), "-Wl,-rpath,$ORIGIN",
    ])


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library (sm_100a only), and the binding's native module."""
    if not force and not is_stale():
        return LIB_PATH
    if force or _stale(LIB_PATH, _deps()):
        cmd = [
            _nvcc(), "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-O3", "-lineinfo", "--threads", "8",
            "-gencode", "arch=compute_100a,code=sm_100a",
            "-I", INCLUDE_DIR, "-I", CSRC,
            "-o", LIB_PATH,
        ] + sources() + ["-lcuda"]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        log = _run(cmd)
        if verbose:
            print(log)
    _build_native()
    return LIB_PATH


if __name__ == "__main__":
    import sys
    print(build_library(force=True, verbose="-v" in sys.argv))
