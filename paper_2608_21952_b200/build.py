"""Builds libssdi8.so (the C-ABI CUDA library) in-tree for sm_100a with nvcc, and _marshal.so (the argument marshalling of
the Python binding) with the host compiler against the installed torch."""
from __future__ import annotations

import glob
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libssdi8.so")
MARSHAL_SRC = os.path.join(CSRC, "marshal.cpp")
MARSHAL = os.path.join(HERE, "_marshal.so")
MARSHAL_STAMP = os.path.join(HERE, "_marshal.built_for")   # the torch build that _marshal.so was compiled against

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17", "--threads", "0",
              "-Xcompiler", "-fPIC", "-shared", "-Xlinker", "-soname=libssdi8.so"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        [os.path.join(os.path.dirname(HERE), "include", "ssdi8.h")]
    return any(os.path.getmtime(p) > t for p in deps)


def build_marshal(force: bool = False) -> str:
    header = os.path.join(os.path.dirname(HERE), "include", "ssdi8.h")
    import sysconfig
    import torch
    built_for = f"torch {torch.__version__}, {sysconfig.get_config_var('SOABI')}"
    try:
        with open(MARSHAL_STAMP) as f:
            same = f.read() == built_for
    except OSError:
        same = False
    if not force and same and os.path.exists(MARSHAL) and \
            os.path.getmtime(MARSHAL) >= max(os.path.getmtime(MARSHAL_SRC), os.path.getmtime(header)):
        return MARSHAL
    from torch.utils.cpp_extension import include_paths, library_paths
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           f'-DSSDI8_TORCH_VERSION="{torch.__version__}"']
    cmd += ["-I" + p for p in (*include_paths(), sysconfig.get_paths()["include"], os.path.join(cuda, "include"))]
    cmd += ["-o", MARSHAL, MARSHAL_SRC]
    cmd += ["-L" + p for p in library_paths()]
    cmd += ["-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10", LIB, "-Wl,-rpath,$ORIGIN"]
    subprocess.run(cmd, check=True)
    with open(MARSHAL_STAMP, "w") as f:
        f.write(built_for)
    return MARSHAL


def build(force: bool = False, verbose: bool = False) -> str:
    lib = build_library(force, verbose)
    build_marshal(force)
    return lib


def build_library(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    # the CUDA runtime is linked statically (nvcc's default), so the library only needs the driver
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + sources()
    subprocess.run(cmd, check=True)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
