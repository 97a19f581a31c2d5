"""Build the C-ABI CUDA library for sm_100a with nvcc and the torch argument marshaller with g++ (no GPU
needed to compile)."""
from __future__ import annotations

import os
import re
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpicospec.so")
MARSHAL_SOURCE = os.path.join(CSRC, "marshal.cpp")
SOURCES = [os.path.join(CSRC, "picospec_api.cu")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden"]


def _deps():
    out = list(SOURCES)
    for root in (CSRC, os.path.join(os.path.dirname(HERE), "include")):
        for f in os.listdir(root):
            if f.endswith((".cuh", ".h", ".cu")):
                out.append(os.path.join(root, f))
    return out


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile libpicospec.so in-tree if it is missing or older than its sources."""
    stale = force or not os.path.exists(LIB)
    if not stale:
        t = os.path.getmtime(LIB)
        stale = any(os.path.getmtime(p) > t for p in _deps())
    if stale:
        nvcc = os.environ.get("NVCC", "nvcc")
        extra = os.environ.get("PICOSPEC_NVCC_FLAGS", "").split()     # e.g. -DPICOSPEC_STAGES_BF16=3
        cmd = [nvcc] + NVCC_FLAGS + extra + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + SOURCES
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed building libpicospec.so")
    build_marshal(force)
    return LIB


def marshal_path() -> str:
    """File of the marshaller for the running Python and the installed torch: it is tied to the binary interface
    of both, so both are in its name and a build for others is never loaded."""
    import torch
    return os.path.join(HERE, "_marshal_torch" + re.sub(r"\W", "_", torch.__version__) + sysconfig.get_config_var("EXT_SUFFIX"))


def build_marshal(force: bool = False) -> str:
    """Compile the marshaller (csrc/marshal.cpp) against the installed torch if it is missing or older than
    its sources."""
    path = marshal_path()
    header = os.path.join(os.path.dirname(HERE), "include", "picospec.h")
    if not force and os.path.exists(path) and all(
            os.path.getmtime(p) <= os.path.getmtime(path) for p in (MARSHAL_SOURCE, header)):
        return path
    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    lib = os.path.join(root, "lib")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}",
           "-I" + os.path.join(root, "include"), "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"),
           "-I" + os.path.join(cuda, "include"), "-I" + sysconfig.get_paths()["include"], MARSHAL_SOURCE, "-o", path,
           "-L" + lib, "-Wl,-rpath," + lib, "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
        raise RuntimeError("g++ failed building the marshaller (csrc/marshal.cpp)")
    return path


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
