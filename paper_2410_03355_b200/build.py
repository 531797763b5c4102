"""Builds the CUDA library in-tree: csrc/*.cu -> paper_2410_03355_b200/liblantern.so (sm_100a), and the native part of the
binding: csrc/call.cpp -> paper_2410_03355_b200/_call.so."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "liblantern.so")
CALL = os.path.join(HERE, "_call.so")

OBJ = os.path.join(HERE, "_build")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xfatbin", "-compress-all"]


def sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cu"))


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(CALL):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(CALL))
    deps = sources() + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    deps += [os.path.join(CSRC, "call.cpp"), os.path.join(ROOT, "include", "lantern.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every kernel for sm_100a with nvcc (one process per translation unit, in parallel:
    the fused kernel's variants sit in files of their own), link; returns the shared library's path."""
    if not force and not _stale():
        return LIB
    from concurrent.futures import ThreadPoolExecutor
    nvcc = os.environ.get("NVCC", "nvcc")
    os.makedirs(OBJ, exist_ok=True)
    common = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
             ["-I", os.path.join(ROOT, "include"), "-I", CSRC]

    def compile_one(src):
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        subprocess.check_call(common + ["-c", src, "-o", obj])
        return obj

    def compile_call():    # (the libraries are torch's, which is imported before it)
        import sysconfig

        import torch
        at = os.path.dirname(torch.__file__)
        inc = os.path.join(at, "include")
        subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "none", "-O2", "-std=c++17",
                               "-Xcompiler", "-fPIC", "-shared",
                               f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                               "-I", os.path.join(ROOT, "include"), "-I", sysconfig.get_paths()["include"], "-I", inc,
                               "-I", os.path.join(inc, "torch", "csrc", "api", "include"),
                               os.path.join(CSRC, "call.cpp"), "-o", CALL, "-L", os.path.join(at, "lib"),
                               "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"])

    with ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as pool:
        call = pool.submit(compile_call)
        objs = list(pool.map(compile_one, sources()))
        call.result()
    subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB] + objs)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
