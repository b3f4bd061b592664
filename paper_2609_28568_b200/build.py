"""Compile the CUDA library in-tree for sm_100a (nvcc cross-compiles without a GPU), and the native half
of its Python binding."""
from __future__ import annotations

import os
import subprocess
import sysconfig

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
_CSRC = os.path.join(_PKG, "csrc")
LIB_PATH = os.path.join(_PKG, "libnb_linear.so")
NATIVE_PATH = os.path.join(_PKG, "_native.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared",
]


def sources() -> list[str]:
    return sorted(os.path.join(_CSRC, f) for f in os.listdir(_CSRC))


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH) or not os.path.exists(NATIVE_PATH):
        return True
    t = min(os.path.getmtime(LIB_PATH), os.path.getmtime(NATIVE_PATH))
    deps = sources() + [os.path.join(_ROOT, "include", "nb_linear.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Build ``libnb_linear.so`` and ``_native.so`` next to the package if they are missing or older than
    their sources."""
    if force or is_stale():
        nvcc = os.environ.get("NVCC", "nvcc")
        cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(_ROOT, "include"), "-I", _CSRC,
               "-o", LIB_PATH, os.path.join(_CSRC, "nb_linear.cu")]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        subprocess.run(cmd, check=True)
        _build_native()
    return LIB_PATH


def _build_native() -> None:
    import torch
    from torch.utils import cpp_extension
    cuda = os.environ.get("CUDA_HOME") or cpp_extension.CUDA_HOME or "/usr/local/cuda"
    inc = [os.path.join(_ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(cuda, "include"),
           *cpp_extension.include_paths()]
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++20", "-fPIC", "-shared",
                    f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                    *[a for i in inc for a in ("-isystem" if "torch" in i else "-I", i)],
                    "-o", NATIVE_PATH, os.path.join(_CSRC, "native.cpp"), "-L", _PKG, "-l:libnb_linear.so",
                    "-Wl,-rpath,$ORIGIN", "-L", lib, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"],
                   check=True)


if __name__ == "__main__":
    print(build(force=True, verbose=True))
