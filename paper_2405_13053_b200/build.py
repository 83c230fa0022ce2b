"""Builds the CUDA library (sm_100a only) with nvcc and the native half of the Python binding with g++, both in-tree; no
GPU is needed to compile."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB_PATH = os.path.join(_PKG, "libmeteora.so")
NATIVE_PATH = os.path.join(_PKG, "_native.so")
NATIVE_SOURCE = "native.cpp"
SOURCES = ["api.cu", "host_copy.cu", "gate_topk.cu", "route.cu", "lora.cu", "gemm_simt.cu", "wgemm_tcgen05.cu", "lora_static.cu",
           "gate_backward.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    built = os.path.getmtime(target)
    deps = [os.path.join(CSRC, f) for f in sources] + [os.path.join(_ROOT, "include", "meteora.h")]
    return any(os.path.getmtime(d) > built for d in deps)


def _build_native(verbose: bool) -> None:
    """csrc/native.cpp -> _native.so, a CPython extension on torch's C++ API that links to libmeteora.so beside it."""
    from torch.utils import cpp_extension

    includes = [os.path.join(_ROOT, "include"), sysconfig.get_paths()["include"], *cpp_extension.include_paths("cuda")]
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", os.path.join(CSRC, NATIVE_SOURCE), "-o", NATIVE_PATH,
           *[flag for d in includes for flag in ("-isystem" if d != includes[0] else "-I", d)],
           *[f"-L{d}" for d in cpp_extension.library_paths("cuda")], f"-L{_PKG}", "-l:libmeteora.so", "-Wl,-rpath,$ORIGIN",
           "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python"]
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or proc.returncode != 0:
        sys.stderr.write(proc.stdout + proc.stderr)
    if proc.returncode != 0:
        raise RuntimeError("g++ failed building _native.so")


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libmeteora.so next to the package, and the native binding beside it; returns the library's path."""
    _build_cuda(force, verbose)
    if force or _stale(NATIVE_PATH, [NATIVE_SOURCE]):
        _build_native(verbose)
    return LIB_PATH


def _build_cuda(force: bool, verbose: bool) -> str:
    if not force and not _stale(LIB_PATH, [f for f in os.listdir(CSRC) if f != NATIVE_SOURCE]):
        return LIB_PATH
    cmd = [_nvcc(), *NVCC_FLAGS, "-I", os.path.join(_ROOT, "include"), "-I", CSRC, "-shared", "-o", LIB_PATH,
           *[os.path.join(CSRC, s) for s in SOURCES]]
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or proc.returncode != 0:
        sys.stderr.write(proc.stdout + proc.stderr)
    if proc.returncode != 0:
        raise RuntimeError("nvcc failed building libmeteora.so")
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
