"""Builds the native code in-tree: the CUDA library with nvcc for sm_100a (no JIT cache is involved)."""
from __future__ import annotations

import glob
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
INCLUDE = os.path.join(_ROOT, "include")
LIB_DIR = os.path.join(_PKG, "_lib")
LIB_PATH = os.path.join(LIB_DIR, "libspechub.so")
BINDING_SRC = os.path.join(CSRC, "native_binding.cpp")
BINDING_PATH = os.path.join(LIB_DIR, "_spechub_native.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
]
LINK_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-cudart", "static"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _headers():
    return glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(INCLUDE, "*.h"))


def _older(path: str, deps) -> bool:
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    return any(os.path.getmtime(f) > t for f in deps)


def is_stale() -> bool:
    return _older(LIB_PATH, sources() + _headers())


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ (in parallel) into one shared library; returns its path."""
    if not force and not is_stale():
        return LIB_PATH
    obj_dir = os.path.join(LIB_DIR, "obj")
    os.makedirs(obj_dir, exist_ok=True)
    nvcc = os.environ.get("NVCC", "nvcc")

    def compile_one(src: str) -> str:
        obj = os.path.join(obj_dir, os.path.basename(src) + ".o")
        if force or _older(obj, [src] + _headers()):
            tmp = obj + ".%d.tmp.o" % os.getpid()
            subprocess.check_call([nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + [
                "-I", INCLUDE, "-I", CSRC, "-c", "-o", tmp, src])
            os.replace(tmp, obj)
        return obj

    with ThreadPoolExecutor(max_workers=max(1, os.cpu_count() or 1)) as pool:
        objs = list(pool.map(compile_one, sources()))
    tmp = LIB_PATH + ".%d.tmp" % os.getpid()
    subprocess.check_call([nvcc] + LINK_FLAGS + ["-o", tmp] + objs)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


def binding_is_stale() -> bool:
    return _older(BINDING_PATH, [BINDING_SRC] + glob.glob(os.path.join(INCLUDE, "*.h")))


def build_binding(force: bool = False) -> str:
    """Compile the CPython module (against this interpreter's torch and ``libspechub.so``); returns its path."""
    if not force and not binding_is_stale():
        return BINDING_PATH
    import sysconfig

    import torch
    from torch.utils import cpp_extension as ext

    build_library()
    include = [sysconfig.get_paths()["include"], INCLUDE] + ext.include_paths("cuda")
    tmp = BINDING_PATH + ".%d.tmp" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
    cmd += [x for i in include for x in ("-isystem", i)] + ["-o", tmp, BINDING_SRC]
    cmd += [x for d in ext.library_paths("cuda") for x in ("-L" + d, "-Wl,-rpath," + d)]
    cmd += ["-L" + LIB_DIR, "-Wl,-rpath,$ORIGIN", "-l:libspechub.so", "-ltorch_python", "-ltorch", "-ltorch_cpu",
            "-ltorch_cuda", "-lc10_cuda", "-lc10"]
    subprocess.check_call(cmd)
    os.replace(tmp, BINDING_PATH)
    return BINDING_PATH


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
    print(build_binding(force=True))
