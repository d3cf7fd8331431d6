"""Build libprecc.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a.

The library is split into several translation units (the attention kernels per head dimension, the
projection kernels, the entry points) that are compiled side by side and linked into one shared object.  Beside it
a small CPython extension (`_native`, csrc/pybind.cpp) is built that turns torch tensors into the arguments of its calls.
"""
from __future__ import annotations

import concurrent.futures
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "build")
LIB = os.path.join(HERE, "libprecc.so")
NATIVE_SRC = os.path.join(CSRC, "pybind.cpp")
NATIVE = os.path.join(HERE, "_native.so")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))
HEADERS = sorted(f for f in os.listdir(CSRC) if f.endswith((".cuh", ".h"))) + [os.path.join("..", "..", "include", "precc.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "--use_fast_math",
              "-Xcompiler", "-fPIC"]


def _newest_header() -> float:
    return max(os.path.getmtime(os.path.join(CSRC, h)) for h in HEADERS)


def _obj(src: str) -> str:
    return os.path.join(OBJ, src[:-3] + ".o")


def resource_log(src: str) -> str:
    """What ptxas reported of the unit's kernels: registers, shared memory, spills."""
    return os.path.join(OBJ, src[:-3] + ".ptxas.log")


def _stale(src: str, hdr_time: float) -> bool:
    o = _obj(src)
    if not os.path.exists(o) or not os.path.exists(resource_log(src)):
        return True
    t = os.path.getmtime(o)
    return os.path.getmtime(os.path.join(CSRC, src)) > t or hdr_time > t


def _compile(nvcc: str, src: str) -> str:
    extra = os.environ.get("PRECC_NVCC_FLAGS", "").split()          # e.g. -DPRECC_PF_TRACE -DPRECC_GEMM_TRACE (timeline stamps)
    cmd = [nvcc] + NVCC_FLAGS + extra + ["-Xptxas=-v", "-c", os.path.join(CSRC, src), "-o", _obj(src)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}{r.stderr}")
    with open(resource_log(src), "w") as f:
        f.write(r.stdout + r.stderr)
    return r.stderr


def _build_native(force: bool):
    """The marshalling extension: host code against torch's headers, linked to libprecc.so next to it."""
    deps = [NATIVE_SRC, os.path.join(HERE, "..", "include", "precc.h")]
    if not force and os.path.exists(NATIVE) and all(os.path.getmtime(d) <= os.path.getmtime(NATIVE) for d in deps):
        return
    import torch
    root = os.path.dirname(torch.__file__)
    lib_dir = os.path.join(root, "lib")
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"], "/usr/local/cuda/include"]
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", NATIVE_SRC,
           "-o", NATIVE] + [f"-I{d}" for d in inc] + [
           LIB, f"-L{lib_dir}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{lib_dir}"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"building {NATIVE} failed:\n{r.stdout}{r.stderr}")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile what is missing or out of date, link, and return the library path."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    os.makedirs(OBJ, exist_ok=True)
    hdr_time = _newest_header()
    todo = [s for s in SOURCES if force or _stale(s, hdr_time)]
    if not todo and os.path.exists(LIB) and all(os.path.getmtime(_obj(s)) <= os.path.getmtime(LIB) for s in SOURCES):
        _build_native(False)
        return LIB
    with concurrent.futures.ThreadPoolExecutor(max_workers=min(len(todo), os.cpu_count() or 1) or 1) as pool:
        for log in pool.map(lambda s: _compile(nvcc, s), todo):
            if verbose:
                sys.stderr.write(log)
    r = subprocess.run([nvcc, "-shared", "-Xlinker", "-soname=libprecc.so", "-o", LIB] + [_obj(s) for s in SOURCES], capture_output=True, text=True)
    if r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
        raise RuntimeError("linking libprecc.so failed")
    _build_native(force)
    return LIB


if __name__ == "__main__":
    print(build(force="-f" in sys.argv, verbose="-v" in sys.argv))
