"""Builds libcachefocus.so in-tree with nvcc for sm_100a, and the native part of its Python binding with g++."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import sysconfig
import warnings
from importlib import metadata

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG_DIR)
LIB_PATH = os.path.join(PKG_DIR, "libcachefocus.so")
# the native part of the binding uses torch's and Python's C++ interfaces: a module built for others is another file
NATIVE_PATH = os.path.join(PKG_DIR, "_native-torch%s-%s.so" % (metadata.version("torch"), sys.implementation.cache_tag))
NATIVE_SOURCE = os.path.join(PKG_DIR, "csrc", "binding.cpp")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "--threads", "0"]


def sources():
    return sorted(glob.glob(os.path.join(PKG_DIR, "csrc", "*.cu")))


def _stale(path, deps) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(p) > os.path.getmtime(path) for p in deps)


def _run(cmd) -> str:
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if proc.returncode != 0:
        raise RuntimeError(os.path.basename(cmd[0]) + " failed:\n" + proc.stdout + proc.stderr)
    return proc.stderr


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source into one shared library; returns its path."""
    headers = glob.glob(os.path.join(ROOT, "include", "*.h"))
    if force or _stale(LIB_PATH, sources() + glob.glob(os.path.join(PKG_DIR, "csrc", "*.cuh")) + headers):
        nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
        cmd = [nvcc] + NVCC_FLAGS + ["-I", os.path.join(ROOT, "include"), "-I", os.path.join(PKG_DIR, "csrc"),
                                     "-o", LIB_PATH] + sources()
        if verbose:
            cmd.insert(1, "-Xptxas=-v")
        log = _run(cmd)
        if verbose:
            print(log)
    if force or _stale(NATIVE_PATH, [NATIVE_SOURCE] + headers):
        try:
            build_native()
        except (RuntimeError, OSError) as e:             # no g++, no torch headers: the binding goes through ctypes
            if os.path.exists(NATIVE_PATH):
                os.remove(NATIVE_PATH)                   # built from other sources
            warnings.warn("the native part of the binding was not built (%s); calls are marshalled by ctypes" % e)
    return LIB_PATH


def build_native() -> None:
    import torch
    torch_dir = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    include = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(cuda, "include"),
               os.path.join(torch_dir, "include"), os.path.join(torch_dir, "include", "torch", "csrc", "api", "include")]
    _run([shutil.which("g++") or "g++", "-O2", "-std=c++17", "-shared", "-fPIC",
          "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch.compiled_with_cxx11_abi()] + ["-I" + i for i in include] +
         [NATIVE_SOURCE, "-o", NATIVE_PATH, "-L" + PKG_DIR, "-l:" + os.path.basename(LIB_PATH), "-Wl,-rpath,$ORIGIN",
          "-L" + os.path.join(torch_dir, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])


if __name__ == "__main__":
    print(build(force=True, verbose=True))
