"""Builds the C-ABI library `libdgq.so` for sm_100a with nvcc and the Python binding's native half
`_native.so` with g++ (both without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "csrc", "dgq.cu")
LIB = os.path.join(HERE, "libdgq.so")
NATIVE_SRC = os.path.join(HERE, "csrc", "binding.cpp")
NATIVE = os.path.join(HERE, "_native.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC,-ffp-contract=off", "-shared",
]


def _sources():
    d = os.path.join(HERE, "csrc")
    out = [os.path.join(d, f) for f in os.listdir(d) if f.endswith((".cu", ".cuh"))]
    out.append(os.path.join(os.path.dirname(HERE), "include", "dgq.h"))
    return out


def _older(target, sources) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(s) > os.path.getmtime(target) for s in sources)


def needs_build() -> bool:
    return _older(LIB, _sources())


def _run(cmd, verbose):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(" ".join(cmd) + " failed:\n" + res.stdout + res.stderr)
    if verbose:
        sys.stderr.write(res.stderr)


def build_native(force: bool = False, verbose: bool = False) -> str:
    """The CPython extension links libdgq.so by its place next to it and torch's libraries by name (torch is imported
    first)."""
    if not force and not _older(NATIVE, [NATIVE_SRC, os.path.join(os.path.dirname(HERE), "include", "dgq.h")]):
        return NATIVE
    import torch
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], "/usr/local/cuda/include"]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *(f"-I{i}" for i in inc), NATIVE_SRC, "-o", NATIVE,
           f"-L{HERE}", "-l:libdgq.so", "-Wl,-rpath,$ORIGIN", f"-L{os.path.join(root, 'lib')}", "-ltorch_python",
           "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    _run(cmd, verbose)
    return NATIVE


def build(force: bool = False, verbose: bool = False) -> str:
    if force or needs_build():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        _run([nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + [SRC, "-o", LIB], verbose)
    build_native(force, verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
