"""Builds the CUDA library (libbittrain.so) in-tree with nvcc for sm_100a, and the extension module
(_pycall) the binding calls it through."""
from __future__ import annotations

import glob
import os
import platform
import shutil
import subprocess
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
INCLUDE = os.path.join(os.path.dirname(PKG_DIR), "include")
LIB_PATH = os.path.join(PKG_DIR, "libbittrain.so")
CALLER_SRC = os.path.join(CSRC, "bt_pycall.c")
CALLER_PATH = os.path.join(PKG_DIR, "_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
AUTOGRAD_SRC = os.path.join(CSRC, "bt_autograd.cpp")
AUTOGRAD_PATH = os.path.join(PKG_DIR, "_autograd" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
AUTOGRAD_BUILT_FOR = os.path.join(PKG_DIR, "_autograd.built_for")      # the torch version that AUTOGRAD_PATH fits

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))


def is_stale(path: str = LIB_PATH) -> bool:
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    return any(os.path.getmtime(p) > t for p in _deps())


def native_calls() -> bool:
    """Is there an extension module for calls on this host?  (It rests on the argument passing of x86-64.)"""
    return platform.machine() == "x86_64"


def build_caller(force: bool = False) -> str:
    """Compile the extension module the binding calls the library through; returns its path."""
    if not native_calls():
        return CALLER_PATH
    if not force and os.path.exists(CALLER_PATH) and os.path.getmtime(CALLER_PATH) >= os.path.getmtime(CALLER_SRC):
        return CALLER_PATH
    tmp = CALLER_PATH + ".tmp%d" % os.getpid()
    subprocess.check_call(["gcc", "-O2", "-Wall", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-o", tmp, CALLER_SRC])
    os.replace(tmp, CALLER_PATH)
    return CALLER_PATH


def autograd_built_for() -> str:
    """The torch version that the extension module of the autograd integration was built for ("" if unknown)."""
    try:
        with open(AUTOGRAD_BUILT_FOR) as f:
            return f.read()
    except FileNotFoundError:
        return ""


def build_autograd(force: bool = False) -> str:
    """Compile the extension module of the autograd integration against torch's C++ headers; returns its path.  It fits the
    torch that it was built for only, whatever the age of the files."""
    import torch
    newest = max(os.path.getmtime(f) for f in (AUTOGRAD_SRC, os.path.join(INCLUDE, "bittrain.h")))
    if not force and os.path.exists(AUTOGRAD_PATH) and os.path.getmtime(AUTOGRAD_PATH) >= newest and autograd_built_for() == torch.__version__:
        return AUTOGRAD_PATH
    from torch.utils import cpp_extension
    headers = cpp_extension.include_paths() + [os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")]
    tmp = AUTOGRAD_PATH + ".tmp%d" % os.getpid()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-shared", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI,
                           "-I", sysconfig.get_paths()["include"], "-I", INCLUDE]
                          + [a for h in headers for a in ("-isystem", h)] + ["-o", tmp, AUTOGRAD_SRC]
                          + ["-L" + d for d in cpp_extension.library_paths()]
                          + ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10_cuda", "-lc10"])
    os.replace(tmp, AUTOGRAD_PATH)
    with open(AUTOGRAD_BUILT_FOR, "w") as f:
        f.write(torch.__version__)
    return AUTOGRAD_PATH


def build_library(force: bool = False, verbose: bool = False, out: str = LIB_PATH, extra_flags=()) -> str:
    """Compile every .cu under csrc/ into one shared object; returns its path.  `out` and
    `extra_flags` (preprocessor defines and the like) are for the checking builds the tests use;
    the product library is the default."""
    if out == LIB_PATH:
        build_caller(force)
        build_autograd(force)
    if not force and not is_stale(out):
        return out
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    os.makedirs(os.path.dirname(out), exist_ok=True)
    tmp = out + ".tmp%d" % os.getpid()
    cmd = [nvcc] + NVCC_FLAGS + list(extra_flags) + (["-Xptxas", "-v"] if verbose else []) + [
        "-I", INCLUDE, "-I", CSRC, "-o", tmp] + sources()
    subprocess.check_call(cmd)
    os.replace(tmp, out)
    return out


if __name__ == "__main__":
    import sys
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
