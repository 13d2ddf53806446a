"""Build the CUDA library in-tree with nvcc for sm_100a.

    python -m paper_2507_17769_b200.build [--force] [--verbose]

Compiles every ``csrc/*.cu`` into ``libpolyserve_attn.so`` next to this file, and ``csrc/pycalls.c`` and ``csrc/torch_calls.cpp``
into the extension modules of the calls of every iteration, with addresses and with torch tensors.  nvcc cross-compiles, so no
GPU is needed to build.  Only the last of the three needs torch, and belongs to the torch that it was built against.
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ_DIR = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libpolyserve_attn.so")
CALLS = os.path.join(HERE, "_pycalls.so")
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xptxas", "-v",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def library_files():
    """What the library and the extension module of the calls through addresses are built from."""
    return sources() + [os.path.join(CSRC, "pycalls.c")] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(HERE, "..", "include", "*.h"))


def torch_calls_path() -> str:
    """The extension module of the calls with tensors, for this interpreter and this torch, whose C++ interface is its own."""
    import torch

    return os.path.join(HERE, "_torch_calls.%s.torch-%s.so" % (sys.implementation.cache_tag, torch.__version__))


def build_torch_calls(force: bool = False, build: bool = True) -> str:
    """Build it if its source is newer or this torch has none (``build=False``: take it as it is)."""
    import torch

    path, src = torch_calls_path(), os.path.join(CSRC, "torch_calls.cpp")
    if not build or (not force and os.path.exists(path) and os.path.getmtime(path) >= os.path.getmtime(src)):
        return path
    root = os.path.dirname(torch.__file__)
    tmp = path + ".tmp.%d" % os.getpid()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
                           "-I", os.path.join(root, "include"), "-I", sysconfig.get_paths()["include"], "-o", tmp, src,
                           "-L", os.path.join(root, "lib"), "-lc10", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, path)
    return path


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(CALLS) and os.path.exists(LIB) and os.path.getmtime(LIB) >= max(map(os.path.getmtime, library_files())):
        return LIB
    os.makedirs(OBJ_DIR, exist_ok=True)
    nvcc = _nvcc()

    def compile_one(src):
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        proc = subprocess.run([nvcc] + NVCC_FLAGS + ["-c", src, "-o", obj], capture_output=True, text=True)
        return src, obj, proc

    objs = []
    with concurrent.futures.ThreadPoolExecutor(max_workers=8) as pool:
        for src, obj, proc in pool.map(compile_one, sources()):
            if verbose or proc.returncode != 0:
                sys.stderr.write(proc.stdout + proc.stderr)
            if proc.returncode != 0:
                raise RuntimeError("nvcc failed on %s" % src)
            objs.append(obj)
    tmp = CALLS + ".tmp.%d" % os.getpid()
    subprocess.check_call(["gcc", "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-o", tmp,
                           os.path.join(CSRC, "pycalls.c")])
    os.replace(tmp, CALLS)
    tmp = LIB + ".tmp.%d" % os.getpid()
    subprocess.check_call([nvcc, "-shared", "-o", tmp] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"])
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
    print(build_torch_calls(force="--force" in sys.argv))
