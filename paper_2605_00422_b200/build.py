"""Builds libbwla.so (the CUDA library behind the C ABI) for sm_100a with nvcc, in-tree.

Usage: ``python -m paper_2605_00422_b200.build [--force] [--verbose]``.
nvcc cross-compiles without a GPU.  The shared object lands beside this file.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libbwla.so")
INCLUDE = os.path.join(_ROOT, "include")
CALLS = os.path.join(_HERE, "_calls.so")   # the native half of the Python binding
OBJ = os.path.join(_HERE, "_build")        # one object per source: an edit recompiles what it touched

NVCC_FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
              "-Xcompiler", "-fPIC", "-shared", "--use_fast_math=false"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _headers():
    return [h for d, e in ((CSRC, "*.cuh"), (CSRC, "*.h"), (INCLUDE, "*.h")) for h in glob.glob(os.path.join(d, e))]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + _headers()
    return any(os.path.getmtime(d) > t for d in deps)


def _newer(path: str, deps) -> bool:
    return os.path.exists(path) and all(os.path.getmtime(d) <= os.path.getmtime(path) for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    build_calls(force)
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")]
    if verbose:
        flags += ["-Xptxas", "-v"]
    os.makedirs(OBJ, exist_ok=True)
    headers = _headers()

    def run(cmd):
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed building libbwla.so")

    def compile_one(src):
        obj = os.path.join(OBJ, os.path.basename(src) + ".o")
        if force or not _newer(obj, [src] + headers):
            run([nvcc] + [f for f in flags if f != "-shared"] + ["-I", INCLUDE, "-I", CSRC, "-c", "-o", obj, src])
        return obj

    with ThreadPoolExecutor(max(2, os.cpu_count() or 2)) as pool:
        objects = list(pool.map(compile_one, sources()))
    run([nvcc] + flags + ["-o", LIB] + objects + ["-lcudart"])
    return LIB


def build_calls(force: bool = False) -> str:
    """csrc/python_calls.cpp against this interpreter's and PyTorch's headers (g++ only)."""
    src = os.path.join(CSRC, "python_calls.cpp")
    if not force and _newer(CALLS, [src, os.path.join(INCLUDE, "bwla.h")]):
        return CALLS
    import sysconfig

    import torch
    troot = os.path.dirname(torch.__file__)
    inc = [INCLUDE, os.path.join(troot, "include"), os.path.join(troot, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], "/usr/local/cuda/include"]
    lib = os.path.join(troot, "lib")
    cmd = (["g++", "-std=c++17", "-O2", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] +
           [f"-I{d}" for d in inc] + ["-o", CALLS, src, f"-L{lib}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
                                      f"-Wl,-rpath,{lib}"])
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed building _calls.so")
    return CALLS


def build_microbench() -> str:
    """The instruction-rate probes (stand-alone programs; not part of the library)."""
    nvcc = os.environ.get("NVCC", "nvcc")
    outs = []
    for name in ("issue_rates", "umma_rates"):
        src = os.path.join(_HERE, "microbench", name + ".cu")
        out = os.path.join(_HERE, "microbench", name)
        res = subprocess.run([nvcc, "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a", "-I", INCLUDE,
                              "-I", CSRC, "-o", out, src], capture_output=True, text=True)
        if res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
            raise RuntimeError("nvcc failed building the microbenchmark " + name)
        outs.append(out)
    return " ".join(outs)


if __name__ == "__main__":
    if "--microbench" in sys.argv:
        print(build_microbench())
    else:
        print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
