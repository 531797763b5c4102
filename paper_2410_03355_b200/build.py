"""Builds the CUDA library in-tree: csrc/*.cu -> paper_2410_03355_b200/liblantern.so (sm_100a), and the native part of the
binding: csrc/call.cpp -> paper_2410_03355_b200/_call.<torch and Python it is for>.so."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings

from .binding import call_path

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblantern.so")

OBJ = os.path.join(HERE, "_build")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xfatbin", "-compress-all"]


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _older(path, deps) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(d) > os.path.getmtime(path) for d in deps)


def _stale() -> bool:
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    return _older(LIB, sources() + headers + [os.path.join(ROOT, "include", "lantern.h")])


def _call_stale() -> bool:
    return _older(call_path(), [os.path.join(CSRC, "call.cpp"), os.path.join(ROOT, "include", "lantern.h")])


def _build_call(nvcc: str) -> None:
    """The native part of the binding, for the torch and the Python that run (its libraries are torch's, which is imported before it).
    The library does without it, and so does the binding: where it cannot be built verify() costs more host time."""
    import torch
    path, at = call_path(), os.path.dirname(torch.__file__)
    if os.path.exists(path):
        os.remove(path)
    inc = os.path.join(at, "include")
    try:
        subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "none", "-O2", "-std=c++17",
                               "-Xcompiler", "-fPIC", "-shared",
                               f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                               "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], "-I", inc,
                               "-I", os.path.join(inc, "torch", "csrc", "api", "include"),
                               os.path.join(CSRC, "call.cpp"), "-o", path, "-L", os.path.join(at, "lib"),
                               "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"])
    except subprocess.CalledProcessError as e:
        warnings.warn(f"{os.path.basename(path)} was not built ({e}): verify() will go through ctypes")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every kernel for sm_100a with nvcc (one process per translation unit, in parallel:
    the fused kernel's variants sit in files of their own), link; returns the shared library's path."""
    from concurrent.futures import ThreadPoolExecutor
    nvcc = os.environ.get("NVCC", "nvcc")
    with ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as pool:
        call = pool.submit(_build_call, nvcc) if force or _call_stale() else None
        if force or _stale():
            os.makedirs(OBJ, exist_ok=True)
            common = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
                     ["-I", os.path.join(ROOT, "include"), "-I", CSRC]

            def compile_one(src):
                obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
                subprocess.check_call(common + ["-c", src, "-o", obj])
                return obj

            objs = list(pool.map(compile_one, sources()))
            subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB] + objs)
        if call is not None:
            call.result()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
