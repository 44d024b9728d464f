"""Builds the CUDA library in-tree, csrc/flop_lib.cu -> libflop_b200.so (sm_100a only), and the native half of the Python
binding, csrc/binding_native.cpp -> _binding_native.<python and torch it is for>.so."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc", "flop_lib.cu")
LIB = os.path.join(HERE, "libflop_b200.so")
NATIVE_SRC = os.path.join(HERE, "csrc", "binding_native.cpp")


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found")


def sources():
    d = os.path.join(HERE, "csrc")
    inc = os.path.join(os.path.dirname(HERE), "include", "flop.h")
    return [os.path.join(d, f) for f in sorted(os.listdir(d)) if f.endswith((".cu", ".cuh"))] + [inc]


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(s) <= t for s in sources())


def native_path() -> str:
    """The module is bound to the C++ interface of one torch and one Python: its name carries both, so that no other loads it."""
    import torch
    return os.path.join(HERE, f"_binding_native.{sys.implementation.cache_tag}-torch-{torch.__version__}.so")


def native_up_to_date() -> bool:
    path = native_path()
    if not os.path.exists(path):
        return False
    t = os.path.getmtime(path)
    return all(os.path.getmtime(p) <= t for p in (NATIVE_SRC, sources()[-1]))


def build_native(force: bool = False) -> str:
    """The module links to libflop_b200.so beside it and to the torch libraries that `import torch` has loaded."""
    path = native_path()
    if not force and native_up_to_date():
        return path
    import torch
    t = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I" + os.path.join(t, "include"), "-I" + os.path.join(t, "include", "torch", "csrc", "api", "include"),
           "-I" + sysconfig.get_paths()["include"], "-I" + os.path.join(cuda, "include"), "-o", path, NATIVE_SRC,
           "-L" + os.path.join(t, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python", "-L" + HERE, "-l:libflop_b200.so",
           "-Wl,-rpath,$ORIGIN"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("building the native binding failed:\n" + r.stdout + r.stderr)
    return path


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and up_to_date():
        build_native()
        return LIB
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-lineinfo",
           "-Xcompiler", "-fPIC", "-shared", "-o", LIB, SRC]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + r.stdout + r.stderr)
    if verbose:
        print(r.stderr)
    build_native(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
