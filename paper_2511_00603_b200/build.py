"""Compiles the CUDA sources of this package into libepara.so (sm_100a only), in-tree.

Each source is compiled to an object file under _build/ (in parallel, only when it or a header changed)
and the objects are linked into the shared library."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libepara.so")
SOURCES = ["epara_api.cu", "kernels_misc.cu", "gemm_simt.cu", "gemm_tc.cu", "gemm_stream.cu", "gemm_swap.cu", "attention.cu", "attention_flash.cu", "policy.cu",
           "selftest.cu"]
# Python side of epara_collect; the file's name carries the interpreter's ABI, another interpreter does not load it
FAST_SRC, FAST_LIB = os.path.join(CSRC, "fastcall.cpp"), os.path.join(HERE, "_fastcall" + sysconfig.get_config_var("EXT_SUFFIX"))
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC"]


def _headers():
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh"))]
    return hs + [os.path.join(HERE, "..", "include", "epara.h")]


def _newer(path: str, deps) -> bool:
    """True when `path` is missing or older than one of deps."""
    if not os.path.exists(path):
        return True
    t = os.path.getmtime(path)
    return any(os.path.getmtime(d) > t for d in deps)


def _stale() -> bool:
    return _newer(LIB, [os.path.join(CSRC, s) for s in SOURCES] + _headers())


def build_fastcall(force: bool = False) -> None:
    """The binding works without it (through ctypes): a machine without Python's headers or a C++ compiler that takes the source goes
    without."""
    include = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(include, "Python.h")) or not (force or _newer(FAST_LIB, [FAST_SRC])):
        return
    for old in (FAST_LIB, os.path.join(os.path.dirname(FAST_LIB), "_fastcall.so")):   # of an older source; without an ABI in its name
        if os.path.exists(old):
            os.remove(old)
    part = f"{FAST_LIB}.{os.getpid()}.part"      # renamed when complete: another process may import it meanwhile
    try:
        r = subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-I", include, FAST_SRC, "-o", part],
                           capture_output=True, text=True)
        failed = f"{r.stdout}{r.stderr}exit status {r.returncode}" if r.returncode != 0 else None
        if failed is None:
            os.replace(part, FAST_LIB)
    except OSError as e:
        failed = str(e)
    if failed is not None:
        sys.stderr.write("fastcall.cpp was not built, answers are collected through ctypes:\n" + failed + "\n")


def build(force: bool = False, verbose: bool = False) -> str:
    build_fastcall(force)
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    hdrs = _headers()

    def compile_one(src: str):
        obj = os.path.join(OBJ, src.replace(".cu", ".o"))
        path = os.path.join(CSRC, src)
        if not force and not verbose and not _newer(obj, [path] + hdrs):
            return obj, ""
        cmd = [nvcc] + (["-Xptxas", "-v"] if verbose else []) + FLAGS + ["-c", path, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n" + r.stdout + r.stderr)
        return obj, r.stderr

    with ThreadPoolExecutor(max_workers=min(len(SOURCES), os.cpu_count() or 1)) as ex:
        results = list(ex.map(compile_one, SOURCES))
    if verbose:
        for _, err in results:
            sys.stderr.write(err)
    r = subprocess.run([nvcc, "-shared", "-o", LIB] + [o for o, _ in results], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n" + r.stdout + r.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
