"""Build step: compile the CUDA library in-tree for sm_100a with nvcc (no GPU needed to compile)."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libsna.so")
TORCH_SOURCE = os.path.join(PKG, "csrc_torch", "sna_autograd.cpp")
TORCH_LIB = os.path.join(PKG, "_sna_torch.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-shared"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cpp")))


def stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.hpp")) + \
        glob.glob(os.path.join(os.path.dirname(PKG), "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or stale():
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + sources()
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    return LIB


def build_torch(force: bool = False) -> str:
    """The autograd function: host code only, against the installed PyTorch, linked to the library beside it."""
    header = os.path.join(os.path.dirname(PKG), "include", "sna.h")
    if not force and os.path.exists(TORCH_LIB) and os.path.getmtime(TORCH_LIB) > max(map(os.path.getmtime, (TORCH_SOURCE, header))):
        return TORCH_LIB
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    tmp = TORCH_LIB + f".tmp{os.getpid()}"
    cuda = os.path.dirname(os.path.dirname(NVCC))
    includes = cpp_extension.include_paths() + [sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    libraries = cpp_extension.library_paths()
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
                           "-DTORCH_API_INCLUDE_EXTENSION_H", "-DTORCH_EXTENSION_NAME=_sna_torch", *(f"-I{i}" for i in includes), TORCH_SOURCE, "-o", tmp,
                           *(f"-L{p}" for p in libraries), "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
                           f"-L{PKG}", "-l:libsna.so", "-Wl,-rpath,$ORIGIN", *(f"-Wl,-rpath,{p}" for p in libraries)])
    os.replace(tmp, TORCH_LIB)
    return TORCH_LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_torch(force="--force" in sys.argv))
