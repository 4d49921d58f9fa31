"""Builds libcovspec.so in-tree with nvcc for sm_100a (no torch extension machinery: the library
is a plain C ABI loaded through ctypes), and the native part of the Python binding with g++ against torch's headers."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcovspec.so")
LIB_DEBUG = os.path.join(HERE, "libcovspec_debug.so")     # the same sources with -DCOVSPEC_DEBUG_BOUNDS
SOURCES = ["covspec.cu"]
BINDING_SOURCE = os.path.join(CSRC, "binding.cpp")


def _newest(paths):
    return max(os.path.getmtime(p) for p in paths)


def binding_path() -> str:
    """The native part of the binding holds to one Python and one torch, which its name gives: another one does not find
    it and builds its own."""
    import torch
    return os.path.join(HERE, f"_binding.{sys.implementation.cache_tag}.torch-{torch.__version__}.so")


def needs_build(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != os.path.basename(BINDING_SOURCE)] + \
           [os.path.join(ROOT, "include", "covspec.h")]
    return _newest(deps) > os.path.getmtime(lib)


def build(force: bool = False, verbose: bool = False, debug_bounds: bool = False) -> str:
    """Builds the library if a source is newer than it.  debug_bounds=True builds the checked variant
    (libcovspec_debug.so): index-driven accesses test their index and report COVSPEC_ERR_BOUNDS.
    The native part of the binding is built too; where that fails (no Python headers) the library is complete without
    it, its calls go through ctypes."""
    if not debug_bounds:
        try:
            build_binding(force)
        except (RuntimeError, OSError) as e:
            sys.stderr.write(f"the native part of the binding was not built, calls will go through ctypes: {e}\n")
    LIB = LIB_DEBUG if debug_bounds else globals()["LIB"]
    if not force and not needs_build(LIB):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-shared", "-Xcompiler", "-fPIC", "-O3", "-std=c++17", "-lineinfo",
           "-gencode", "arch=compute_100a,code=sm_100a",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    if debug_bounds:
        cmd.insert(1, "-DCOVSPEC_DEBUG_BOUNDS")
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("nvcc failed building " + os.path.basename(LIB))
    if verbose:
        sys.stderr.write(res.stderr)
    return LIB


def build_binding(force: bool = False) -> str:
    import torch
    target = binding_path()
    if not force and os.path.exists(target) and os.path.getmtime(BINDING_SOURCE) <= os.path.getmtime(target):
        return target
    base = os.path.dirname(torch.__file__)
    libs = os.path.join(base, "lib")
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-shared", "-fPIC", "-std=c++17",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(base, "include"), "-I", os.path.join(base, "include", "torch", "csrc", "api", "include"),
           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"),
           "-o", target, BINDING_SOURCE, "-L", libs, "-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu", "-ltorch_python",
           "-Wl,-rpath," + libs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed building " + os.path.basename(target))
    return target


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv, debug_bounds="--debug-bounds" in sys.argv))
