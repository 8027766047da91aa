"""Builds the CUDA library (libogq.so) in-tree with nvcc for sm_100a.

Every .cu file is compiled to an object of its own (in parallel, and only when it or a header is
newer than the object), then the objects are linked into the shared library.  The CPython module with
the data-path calls (_native, which loads the library itself) is compiled next to it with g++.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
OBJ_DIR = os.path.join(_HERE, "_build")
LIB_PATH = os.path.join(_HERE, "libogq.so")
NATIVE_SRC = os.path.join(CSRC, "ogq_python.cpp")
NATIVE_PATH = os.path.join(_HERE, "_native" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-lineinfo", "-O3", "-std=c++17", "-fmad=false", "--extended-lambda",
    "-Xcompiler", "-fPIC",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _headers():
    return glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + [
        os.path.join(_HERE, "..", "include", "ogq.h")]


def _obj(src: str) -> str:
    return os.path.join(OBJ_DIR, os.path.basename(src)[:-3] + ".o")


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def needs_build() -> bool:
    return _stale(LIB_PATH, sources() + _headers()) or _stale(NATIVE_PATH, [NATIVE_SRC])


def build_native(force: bool = False) -> str:
    if force or _stale(NATIVE_PATH, [NATIVE_SRC]):
        subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                        "-I", sysconfig.get_paths()["include"], NATIVE_SRC, "-o", NATIVE_PATH], check=True)
    return NATIVE_PATH


def build(force: bool = False, verbose: bool = False) -> str:
    build_native(force)
    if not force and not needs_build():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ_DIR, exist_ok=True)
    hdrs = _headers()
    todo = [s for s in sources() if force or _stale(_obj(s), [s] + hdrs)]

    def compile_one(src):
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", _obj(src)]
        return subprocess.run(cmd, check=True, capture_output=True, text=True)

    with ThreadPoolExecutor(max_workers=max(1, min(len(todo), os.cpu_count() or 1))) as pool:
        for res in pool.map(compile_one, todo):
            if verbose:
                print(res.stderr, end="")
    objs = [_obj(s) for s in sources()]
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB_PATH] + objs + ["-ldl"], check=True)
    return LIB_PATH


if __name__ == "__main__":
    import sys

    print(build(force="-f" in sys.argv, verbose="-v" in sys.argv))
