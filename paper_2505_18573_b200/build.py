"""Build ``libe3.so`` (the C-ABI CUDA library, nvcc for sm_100a) and ``_native.so`` (its Python binding) in-tree.

Run as ``python -m paper_2505_18573_b200.build`` or call :func:`build`.  Each is rebuilt when any of its sources or headers is
newer than the binary.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
_CSRC = os.path.join(_PKG, "csrc")
LIB_PATH = os.path.join(_PKG, "libe3.so")
NATIVE_PATH = os.path.join(_PKG, "_native.so")
_NATIVE_SRC = os.path.join(_CSRC, "py", "e3_py.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def sources():
    return sorted(glob.glob(os.path.join(_CSRC, "*.cu")) + glob.glob(os.path.join(_CSRC, "*.cpp")))


def _headers():
    return glob.glob(os.path.join(_CSRC, "*.cuh")) + glob.glob(os.path.join(_CSRC, "*.h")) + glob.glob(os.path.join(_ROOT, "include", "*.h"))


def _older(path: str, deps) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(f) > os.path.getmtime(path) for f in deps)


def needs_build() -> bool:
    return _older(LIB_PATH, sources() + _headers())


def _native_command(out: str):
    import torch
    from torch.utils import cpp_extension
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", os.path.join(_ROOT, "include"), "-I", _CSRC, "-I", sysconfig.get_paths()["include"],
           "-I", os.path.join(cuda, "include")]
    for d in cpp_extension.include_paths():
        cmd += ["-isystem", d]
    cmd += ["-o", out, _NATIVE_SRC, "-L", _PKG, "-l:libe3.so", "-Wl,-rpath,$ORIGIN"]
    for d in cpp_extension.library_paths():
        cmd += ["-L", d]
    # symbols of the CUDA runtime are found in the copy torch has loaded
    return cmd + ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda"]


def build(force: bool = False, verbose: bool = False) -> str:
    def run(cmd, path):
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        subprocess.run(cmd, check=True)
        os.replace(cmd[cmd.index("-o") + 1], path)

    if force or needs_build():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        tmp = LIB_PATH + f".{os.getpid()}.tmp"
        cmd = [nvcc] + (["-Xptxas=-v"] if verbose else []) + NVCC_FLAGS
        run(cmd + ["-I", os.path.join(_ROOT, "include"), "-I", _CSRC, "-o", tmp] + sources(), LIB_PATH)
    if force or _older(NATIVE_PATH, [_NATIVE_SRC] + _headers()):
        run(_native_command(NATIVE_PATH + f".{os.getpid()}.tmp"), NATIVE_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
