"""Builds, in-tree, libs2a.so (the C-ABI library of include/s2a.h, nvcc for sm_100a) and _s2a_torch.so (the
hot half of the Python binding, g++ against torch's headers, linked to libs2a.so beside it)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libs2a.so")
SOURCES = ["api.cu", "fwd_kernel.cu", "bwd_kernels.cu"]
HEADERS = ["host_plan.h", "s2a_params.h", "sm100_ptx.cuh", os.path.join("..", "..", "include", "s2a.h")]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
]
TORCH_LIB = os.path.join(PKG, "_s2a_torch.so")
TORCH_SOURCE = os.path.join(CSRC, "torch_binding.cpp")


def _newest(paths):
    return max(os.path.getmtime(p) for p in paths)


def build(force: bool = False, verbose: bool = False) -> str:
    srcs = [os.path.join(CSRC, s) for s in SOURCES]
    deps = srcs + [os.path.join(CSRC, h) for h in HEADERS]
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest(deps):
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, *NVCC_FLAGS, "-shared", "-o", LIB, *srcs]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
        print(" ".join(cmd), file=sys.stderr)
    subprocess.run(cmd, check=True, cwd=CSRC)
    return LIB


def _built_for(path: str) -> str | None:
    try:
        with open(path) as f:
            return f.read()
    except OSError:
        return None


def build_torch(force: bool = False) -> str:
    import torch

    # a module that was built for another torch or Python would be loaded all the same and misread this one's objects
    stamp, wanted = TORCH_LIB + ".built_for", f"torch {torch.__version__}, python {sys.version}"
    deps = [TORCH_SOURCE, os.path.join(PKG, "..", "include", "s2a.h")]
    if not force and _built_for(stamp) == wanted and os.path.exists(TORCH_LIB) and os.path.getmtime(TORCH_LIB) >= _newest(deps):
        return TORCH_LIB
    root = os.path.join(os.path.dirname(os.path.abspath(torch.__file__)))
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    include = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
               os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-DTORCH_EXTENSION_NAME=_s2a_torch",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DS2A_TORCH_VERSION="{torch.__version__}"', *(f"-I{d}" for d in include), TORCH_SOURCE,
           "-o", TORCH_LIB, f"-L{os.path.join(root, 'lib')}", f"-L{os.path.join(cuda, 'lib64')}", f"-L{PKG}", "-l:libs2a.so",
           "-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-lcudart", "-Wl,-rpath,$ORIGIN"]
    subprocess.run(cmd, check=True)
    with open(stamp, "w") as f:
        f.write(wanted)
    return TORCH_LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
    print(build_torch(force="--force" in sys.argv))
