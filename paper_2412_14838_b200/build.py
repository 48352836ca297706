"""Build libdkv.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _dkv_pycall.so (the native half of
binding.py: argument conversion; only where torch is installed, whose libraries it is linked with) with the host compiler.

``python -m paper_2412_14838_b200.build`` or ``build()``; nvcc cross-compiles without a GPU.
"""
from __future__ import annotations

import importlib.metadata
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdkv.so")
SOURCES = ["dkv.cu"]
PYCALL = os.path.join(HERE, "_dkv_pycall.so")
PYCALL_TORCH = PYCALL + ".torch"        # beside it: the torch version it was linked with
PYCALL_SOURCE = os.path.join(CSRC, "pycall.cpp")
HEADER = os.path.join(os.path.dirname(HERE), "include", "dkv.h")


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: libdkv.so cannot be built")


def torch_version() -> str | None:
    """The installed torch's version, None where there is none (without importing it, which takes seconds)."""
    try:
        return importlib.metadata.version("torch")
    except importlib.metadata.PackageNotFoundError:
        return None


def pycall_built_for() -> str | None:
    """The torch version that _dkv_pycall.so was linked with, if its build left a note."""
    try:
        with open(PYCALL_TORCH) as f:
            return f.read().strip()
    except FileNotFoundError:
        return None


def _stale(lib: str, deps) -> bool:
    return not os.path.exists(lib) or any(os.path.getmtime(d) > os.path.getmtime(lib) for d in deps)


def _run(cmd, verbose: bool) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{os.path.basename(cmd[0])} failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stdout + res.stderr)


def _build_pycall(verbose: bool) -> None:
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), sysconfig.get_paths()["include"], "/usr/local/cuda/include"]
    _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
          f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", *(f"-I{d}" for d in inc), PYCALL_SOURCE,
          "-o", PYCALL, f"-L{HERE}", "-l:libdkv.so", f"-L{root}/lib", "-ltorch_python", "-lc10", "-lc10_cuda",
          "-Wl,-rpath,$ORIGIN", f"-Wl,-rpath,{root}/lib"], verbose)
    with open(PYCALL_TORCH, "w") as f:
        f.write(torch_version() + "\n")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile what is older than its sources, or linked with another torch; return the library's path."""
    kernels = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f != os.path.basename(PYCALL_SOURCE)]
    if force or _stale(LIB, kernels + [HEADER]):
        # uncompressed: unpacking the device code takes the first dkv_create of a process 7 ms and more (10 -> 17-30)
        _run([_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "--no-compress", "-Xptxas", "-v" if verbose else "-O3",
              "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES], verbose)
    if torch_version() and (force or _stale(PYCALL, [PYCALL_SOURCE, HEADER]) or pycall_built_for() != torch_version()):
        _build_pycall(verbose)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
