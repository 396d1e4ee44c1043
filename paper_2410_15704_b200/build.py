"""Build the CUDA library (nvcc, sm_100a) and its Python call path (g++) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LIB = os.path.join(HERE, "librvq_b200.so")
NATIVE = os.path.join(HERE, "_native.so")
SOURCES = sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")))
BINDING = os.path.join(HERE, "csrc", "binding.cpp")
PUBLIC = sorted(glob.glob(os.path.join(ROOT, "include", "*.h")))
HEADERS = sorted(glob.glob(os.path.join(HERE, "csrc", "*.cuh"))) + PUBLIC

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "--threads", "0",
              "-Xcompiler", "-fPIC", "-shared", "-Xlinker", "-soname=librvq_b200.so", "-I" + os.path.join(ROOT, "include")]


def stale(target: str, sources) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in sources)


def build_binding() -> None:
    """_native.so: csrc/binding.cpp against the installed torch's headers."""
    import torch
    from torch.utils import cpp_extension

    libdir = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = cpp_extension.include_paths() + [os.path.join(cuda, "include"), sysconfig.get_paths()["include"],
                                               os.path.join(ROOT, "include")]
    cmd = (["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)] + ["-isystem" + p for p in include] +
           [BINDING, "-o", NATIVE, "-L" + HERE, "-lrvq_b200", "-L" + libdir, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
            "-Wl,-rpath,$ORIGIN"])
    subprocess.check_call(cmd)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into librvq_b200.so and the binding beside it (no GPU needed)."""
    if force or stale(LIB, SOURCES + HEADERS):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + SOURCES + ["-o", LIB]
        subprocess.check_call(cmd)
    if force or stale(NATIVE, [BINDING] + PUBLIC):
        build_binding()
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
