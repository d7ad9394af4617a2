"""Compile the CUDA library in-tree for sm_100a with nvcc (no JIT cache, no torch extension)."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libdivision.so")
NATIVE_SRC = os.path.join(CSRC, "native.cpp")
NATIVE_PATH = os.path.join(PKG_DIR, "_native.so")        # the calls on torch tensors, linked against the library
OBJ_DIR = os.path.join(PKG_DIR, "_build")
SOURCES = ["division.cu", "cluster.cu", "planeshare.cu", "park.cu"]
HEADERS = ["common.cuh", "cluster_plan.cuh", "halves.cuh", "park_plan.cuh", "twopass.cuh", "decompress.cuh", "fused.cuh", "fused_v.cuh", "lagged.cuh", "staged.cuh", "planes.cuh", "planegroup.cuh", "masks.cuh", "lines.cuh", "volume.cuh", os.path.join("..", "..", "include", "division.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-lineinfo", "-std=c++17",
    "-Xcompiler", "-fPIC",
    "--fmad=false",          # one rounding per operation is part of the output contract
    "-Xptxas", "-v",
]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the CUDA library cannot be built")
    return exe


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(NATIVE_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = [os.path.join(CSRC, f) for f in SOURCES + HEADERS]
    return any(os.path.getmtime(d) > t for d in deps) or os.path.getmtime(NATIVE_SRC) > os.path.getmtime(NATIVE_PATH)


def build(force: bool = False, verbose: bool = False) -> str:
    """Build libdivision.so next to this file; returns its path."""
    if not force and not is_stale():
        return LIB_PATH
    os.makedirs(OBJ_DIR, exist_ok=True)
    newest_header = max(os.path.getmtime(os.path.join(CSRC, h)) for h in HEADERS)

    def compile_one(src):
        path, obj = os.path.join(CSRC, src), os.path.join(OBJ_DIR, src[:-3] + ".o")
        log = obj[:-2] + ".log"
        if force or not (os.path.exists(obj) and os.path.getmtime(obj) > max(newest_header, os.path.getmtime(path))):
            _run([_nvcc()] + NVCC_FLAGS + ["-c", path, "-o", obj], verbose, log)
        return obj, log

    with ThreadPoolExecutor(len(SOURCES)) as pool:          # one nvcc per source, side by side
        done = list(pool.map(compile_one, SOURCES))
    _run([_nvcc(), "-shared"] + NVCC_FLAGS[:2] + [obj for obj, _ in done] + ["-o", LIB_PATH], verbose, None)
    _build_native(verbose)
    with open(os.path.join(PKG_DIR, "ptxas_info.log"), "w") as f:
        f.write("".join(open(log).read() for _, log in done))
    return LIB_PATH


def _build_native(verbose):
    """The CPython extension: host C++ only, needs torch's headers and libraries."""
    import sysconfig

    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    includes = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    _run([shutil.which("g++") or "g++", "-O2", "-std=c++17", "-shared", "-fPIC",
          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"] + ["-I" + i for i in includes] +
         [NATIVE_SRC, "-o", NATIVE_PATH, "-L" + os.path.join(root, "lib"), "-L" + PKG_DIR, "-ltorch_python", "-ltorch_cpu", "-lc10",
          "-lc10_cuda", "-l:libdivision.so", "-Wl,-rpath,$ORIGIN"], verbose, None)


def _run(cmd, verbose, log):
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or proc.returncode != 0:
        sys.stderr.write(proc.stdout + proc.stderr)
    if proc.returncode != 0:
        raise RuntimeError("building the library failed: " + os.path.basename(cmd[0]))
    if log:
        with open(log, "w") as f:
            f.write(proc.stderr)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
