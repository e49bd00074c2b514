"""Builds libfgmp.so (sm_100a only) and the CPython entry points _fgmp_torch.so in-tree.  Run as a module or call build()."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
import tempfile
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libfgmp.so")
EXT = os.path.join(HERE, "_fgmp_torch.so")

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target: str, deps: list[str]) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def is_stale() -> bool:
    header = os.path.join(ROOT, "include", "fgmp.h")
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + [header]) or \
        _older(EXT, [os.path.join(CSRC, "fgmp_torch.cpp"), header])


def _build_extension() -> None:
    import torch
    from torch.utils import cpp_extension
    tlib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [sysconfig.get_paths()["include"], os.path.join(ROOT, "include"), os.path.join(cuda, "include")] + cpp_extension.include_paths()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", "-DUSE_C10D_NCCL=0"] +
                          [x for d in inc for x in ("-isystem", d)] +
                          ["-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), os.path.join(CSRC, "fgmp_torch.cpp"),
                           "-o", EXT, "-L", HERE, "-l:libfgmp.so", "-L", tlib, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10",
                           "-lc10_cuda", "-Wl,--no-as-needed", "-ltorch_cuda", "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + tlib])


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not is_stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    with tempfile.TemporaryDirectory() as tmp:
        def compile_one(src: str) -> str:
            obj = os.path.join(tmp, os.path.basename(src) + ".o")
            subprocess.check_call([nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) +
                                  ["-I", os.path.join(ROOT, "include"), "-I", CSRC, "-c", src, "-o", obj])
            return obj
        with ThreadPoolExecutor(os.cpu_count() or 4) as pool:
            objs = list(pool.map(compile_one, sources()))
        subprocess.check_call([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-shared", "-o", LIB] + objs)
    _build_extension()
    return LIB


if __name__ == "__main__":
    build(force=True, verbose="-v" in sys.argv)
    print(LIB)
