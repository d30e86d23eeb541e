"""Build the CUDA library and the binding's marshalling module in-tree (nvcc for sm_100a cross-compiles without a GPU)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcalidrop.so")
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")
HEADER = os.path.join(os.path.dirname(HERE), "include", "calidrop.h")

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-Xcompiler", "-fPIC", "-shared", "--expt-relaxed-constexpr",
]


def marshal_path() -> str:
    """The marshalling module, named after the Python and the torch whose binary interfaces it is compiled against, so
    that a module built for others is never loaded."""
    import torch

    return os.path.join(HERE, f"_marshal.{sys.implementation.cache_tag}-torch{torch.__version__}.so")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        [HEADER]


def _older(target, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(f) > t for f in deps)


def is_stale() -> bool:
    return _older(LIB, _deps()) or _older(marshal_path(), [MARSHAL_SRC, HEADER])


def _build_marshal() -> None:
    import torch
    from torch.utils import cpp_extension

    target = marshal_path()
    tmp = target + f".{os.getpid()}.tmp"
    libs = cpp_extension.library_paths("cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f"-I{sysconfig.get_paths()['include']}"]
    cmd += [f"-isystem{p}" for p in cpp_extension.include_paths("cuda")]
    cmd += ["-o", tmp, MARSHAL_SRC] + [f"-L{p}" for p in libs] + \
        ["-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-ldl"]
    subprocess.check_call(cmd)
    os.replace(tmp, target)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _older(marshal_path(), [MARSHAL_SRC, HEADER]):
        _build_marshal()
    if not force and not _older(LIB, _deps()):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + sources()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
