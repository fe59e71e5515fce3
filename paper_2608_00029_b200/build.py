"""Builds libnova_attn.so in-tree with nvcc for sm_100a (cross-compiles without a GPU), and its Python binding
(_binding.so, host code against the installed torch) with g++."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnova_attn.so")
SOURCES = ["api.cu", "attn_fwd.cu", "attn_bwd.cu", "attn_bwd_pre.cu", "attn_dq.cu", "attn_dq64.cu", "attn_dkdv.cu", "attn_dkdv64.cu",
           "attn_bwd_static.cu", "lmhead.cu", "lmhead_rows.cu"]
BINDING = os.path.join(HERE, "_binding.so")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared", "-cudart", "shared", "-Xlinker", "-soname=libnova_attn.so"]


def _sources():
    return [os.path.join(CSRC, s) for s in SOURCES if os.path.exists(os.path.join(CSRC, s))]


def _built_for() -> str:
    import torch
    return f"torch {torch.__version__}, Python {sys.version_info.major}.{sys.version_info.minor}"


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(BINDING):
        return True
    with open(BINDING, "rb") as f:
        if f"nova binding for {_built_for()}\0".encode() not in f.read():
            return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(BINDING))
    deps = _sources() + [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".h", ".cuh", ".cpp"))]
    deps.append(os.path.join(os.path.dirname(HERE), "include", "nova_attn.h"))
    deps.append(os.path.join(os.path.dirname(HERE), "include", "nova_lmhead.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def _build_binding() -> None:
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    inc = cpp_extension.include_paths() + [sysconfig.get_paths()["include"], "/usr/local/cuda/include"]
    tmp = BINDING + f".tmp{os.getpid()}"
    subprocess.check_call(
        [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
         f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DNOVA_BUILT_FOR="{_built_for()}"'] + [f"-I{p}" for p in inc] +
        ["-o", tmp, os.path.join(CSRC, "binding.cpp"), LIB, f"-L{lib}", "-lc10", "-lc10_cuda", "-ltorch_cpu",
         "-ltorch_python", "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{lib}"])
    os.replace(tmp, BINDING)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source of the library into one shared object; returns its path."""
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + _sources()
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    _build_binding()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
