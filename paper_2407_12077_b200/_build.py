"""Builds libgfwkv6.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the binding's C++ part with g++."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sysconfig
import warnings

import torch

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
LIB_PATH = os.path.join(_PKG, "libgfwkv6.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "--expt-relaxed-constexpr",
]

# Python and torch headers are not a stable interface: the file carries their versions
BINDING_SRC = os.path.join(CSRC, "binding.cpp")
BINDING_PATH = os.path.join(_PKG, f"_binding-{sysconfig.get_config_var('SOABI')}-torch{torch.__version__}.so")


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the gf_wkv6 CUDA library cannot be built")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    deps = glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(_ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def binding_is_stale() -> bool:
    return not os.path.exists(BINDING_PATH) or os.path.getmtime(BINDING_SRC) > os.path.getmtime(BINDING_PATH)


def build_binding(force: bool = False) -> str | None:
    """Compile the binding's C++ part (None where that cannot be done: no compiler or header for it, a compiler that fails, a
    directory that cannot be written.  The Python code does without)."""
    if not force and not binding_is_stale():
        return BINDING_PATH
    gxx, py = shutil.which("g++"), sysconfig.get_paths()["include"]
    inc = os.path.join(os.path.dirname(torch.__file__), "include")
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    if gxx is None or not os.path.exists(os.path.join(py, "Python.h")) or not os.path.exists(inc) or not os.access(_PKG, os.W_OK):
        return None
    tmp = f"{BINDING_PATH}.{os.getpid()}"
    cmd = [gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           "-I", py, "-I", inc, "-I", os.path.join(inc, "torch", "csrc", "api", "include"), "-I", os.path.join(cuda, "include"), "-o", tmp, BINDING_SRC,
           "-L", os.path.join(os.path.dirname(torch.__file__), "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    try:
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode == 0:
            os.replace(tmp, BINDING_PATH)
            return BINDING_PATH
        why = res.stdout + res.stderr
    except OSError as e:
        why = str(e)
    if os.path.exists(tmp):
        os.remove(tmp)
    warnings.warn("the binding's C++ part could not be built (calls go through Python, a few microseconds slower):\n" + why[-2000:], RuntimeWarning)
    return None


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source into libgfwkv6.so, and the binding's C++ part.  Cross-compiles without a GPU."""
    if force or is_stale():
        build_library(verbose)
    build_binding(force)
    return LIB_PATH


def build_library(verbose: bool = False) -> str:
    """Compile every CUDA source into libgfwkv6.so."""
    cmd = [_nvcc(), *NVCC_FLAGS, "-I", os.path.join(_ROOT, "include"), "-I", CSRC,
           "-o", LIB_PATH, *sources()]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    if verbose:
        print(res.stderr)
    return LIB_PATH


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
