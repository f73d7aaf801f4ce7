"""Builds libvispec.so (the C-ABI CUDA library, nvcc for sm_100a) and _native.so (its CPython face, g++) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libvispec.so")
NATIVE_SRC = os.path.join(CSRC, "binding_native.cpp")
NATIVE = os.path.join(HERE, "_native.so")
SOURCES = ["vispec_api.cu", "tree_kernels.cu", "attn_generic.cu", "attn_tc5.cu", "attn_tc5_wide.cu", "attn_static.cu", "accept_sampled.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--use_fast_math", "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def _stale() -> bool:
    header = os.path.join(ROOT, "include", "vispec.h")
    cuda = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h"))]

    def older(target, deps):
        return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)

    return older(LIB, cuda + [header]) or older(NATIVE, [NATIVE_SRC, header])


def _build_native(verbose: bool) -> None:
    """The CPython face: torch's headers give it device pointers and the current stream; it links libvispec.so beside it."""
    import torch
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(ROOT, "include"), "-isystem", sysconfig.get_paths()["include"], "-isystem", inc,
           "-isystem", os.path.join(inc, "torch", "csrc", "api", "include"), "-isystem", cuda, NATIVE_SRC, "-o", NATIVE,
           LIB, "-L", lib, "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError("g++ failed on binding_native.cpp")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu of the library and link them into one shared object, then the CPython face.  Returns the
    library's path."""
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    objs = []
    for src in SOURCES:
        obj = os.path.join(CSRC, src.replace(".cu", ".o"))
        cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c",
               os.path.join(CSRC, src), "-o", obj]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}")
        objs.append(obj)
    # cudart is linked statically (nvcc default); the soname lets the CPython face find the library beside itself
    cmd = [nvcc, "-shared", "-Xlinker", "-soname=libvispec.so", "-o", LIB, *objs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("link failed")
    _build_native(verbose)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
