"""Builds libsplash_mla.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the extension module that
takes torch tensors to it."""
from __future__ import annotations

import glob
import os
import re
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsplash_mla.so")
TORCH_SRC = os.path.join(CSRC, "splash_torch.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden", "--use_fast_math",
    "-shared",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def torch_ext_path() -> str:
    """The extension module for the torch in use.  Its version is part of the name: a module built against another one has other
    C++ interfaces, and neither counts as built nor is loaded."""
    import torch
    return os.path.join(HERE, "_splash_torch.torch_" + re.sub(r"[^0-9A-Za-z]+", "_", torch.__version__) + ".so")


def _older(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _headers():
    return glob.glob(os.path.join(HERE, "..", "include", "*.h"))


def _build_torch_ext() -> None:
    """The extension is a host file against torch's C++ headers; it finds the library beside it and torch's libraries
    in the process (the package imports torch first)."""
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    flags = ["-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
             f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}"]
    for path in cpp_extension.include_paths() + [sysconfig.get_paths()["include"], "/usr/local/cuda/include"]:
        flags += ["-isystem", path]
    libs = ["-L" + HERE, "-lsplash_mla"]
    for path in cpp_extension.library_paths():
        libs.append("-L" + path)
    libs += ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN"]
    target = torch_ext_path()
    subprocess.check_call([os.environ.get("CXX", "g++")] + flags + ["-o", target, TORCH_SRC] + libs)
    for other in glob.glob(os.path.join(HERE, "_splash_torch*.so")):      # of another torch, or of the time before versions had names
        if other != target:
            os.remove(other)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers()):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + sources()
        subprocess.check_call(cmd)
    if force or _older(torch_ext_path(), [TORCH_SRC] + _headers()):
        _build_torch_ext()
    return LIB


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose="-v" in sys.argv)
    print(LIB)
