"""Build the CUDA library in-tree with nvcc for sm_100a.

    python -m paper_2507_17769_b200.build [--force] [--verbose]

Compiles every ``csrc/*.cu`` into ``libpolyserve_attn.so`` next to this file, and ``csrc/pycalls.c`` and ``csrc/torch_calls.cpp``
into the extension modules of the calls of every iteration, with addresses and with torch tensors.  nvcc cross-compiles, so no
GPU is needed to build.
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
TORCH_CALLS = os.path.join(HERE, "_torch_calls.so")
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


def _deps_mtime() -> float:
    files = sources() + [os.path.join(CSRC, "pycalls.c"), os.path.join(CSRC, "torch_calls.cpp")] + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(HERE, "..", "include", "*.h"))
    return max(os.path.getmtime(f) for f in files)


def _build_torch_calls():
    import torch

    root = os.path.dirname(torch.__file__)
    tmp = TORCH_CALLS + ".tmp.%d" % os.getpid()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
                           "-I", os.path.join(root, "include"), "-I", sysconfig.get_paths()["include"], "-o", tmp, os.path.join(CSRC, "torch_calls.cpp"),
                           "-L", os.path.join(root, "lib"), "-lc10", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, TORCH_CALLS)


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and os.path.exists(CALLS) and os.path.exists(TORCH_CALLS) and os.path.exists(LIB) and os.path.getmtime(LIB) >= _deps_mtime():
        return LIB
    os.makedirs(OBJ_DIR, exist_ok=True)
    nvcc = _nvcc()

    def compile_one(src):
        obj = os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")
        proc = subprocess.run([nvcc] + NVCC_FLAGS + ["-c", src, "-o", obj], capture_output=True, text=True)
        return src, obj, proc

    objs = []
    with concurrent.futures.ThreadPoolExecutor(max_workers=8) as pool:
        torch_calls = pool.submit(_build_torch_calls)
        for src, obj, proc in pool.map(compile_one, sources()):
            if verbose or proc.returncode != 0:
                sys.stderr.write(proc.stdout + proc.stderr)
            if proc.returncode != 0:
                raise RuntimeError("nvcc failed on %s" % src)
            objs.append(obj)
        torch_calls.result()
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
