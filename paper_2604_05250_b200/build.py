"""Builds in-tree: csrc/*.cu -> libdualdiff.so (sm_100a only), csrc/host_call.cpp -> _host_call-*.so (the
native host side of the Python calls; one file per Python and torch version)."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdualdiff.so")
HOST_SRC = os.path.join(CSRC, "host_call.cpp")
LIB_CHECK = os.path.join(HERE, "libdualdiff_check.so")      # the same sources with -DDD_BOUNDS_CHECK

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-lineinfo",
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-Xcompiler", "-fPIC", "-shared", "-cudart", "static",
]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA library cannot be built")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(lib=None) -> bool:
    lib = lib or LIB
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(HERE, "..", "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    if force or _stale():
        cmd = [_nvcc(), *NVCC_FLAGS, *extra_flags, "-o", LIB, *sources()]
        if verbose:
            print(" ".join(cmd), flush=True)
        subprocess.run(cmd, check=True)
    build_host(force, verbose)
    return LIB


def host_path() -> str:
    """The native host side for this Python and this torch (a module built against another one is not loaded)."""
    import torch
    return os.path.join(HERE, f"_host_call-{sys.implementation.cache_tag}-torch{torch.__version__}.so")


def build_host(force: bool = False, verbose: bool = False):
    """The module behind binding.py's calls on device tensors: torch's headers and libraries, no CUDA code.  Where it
    cannot be built (no C++ compiler, no headers) a warning is given: the Python form serves every call."""
    import torch
    host = host_path()
    if force or not os.path.exists(host) or os.path.getmtime(host) < os.path.getmtime(HOST_SRC):
        import sysconfig
        import warnings
        root = os.path.dirname(torch.__file__)
        try:
            cuda = os.path.dirname(os.path.dirname(_nvcc()))
            cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
                   "-I" + os.path.join(root, "include"), "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"),
                   "-I" + os.path.join(cuda, "include"), "-I" + sysconfig.get_paths()["include"],
                   "-o", host, HOST_SRC, "-L" + os.path.join(root, "lib"),
                   "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda"]
            if verbose:
                print(" ".join(cmd), flush=True)
            subprocess.run(cmd, check=True)
        except (OSError, RuntimeError, subprocess.CalledProcessError) as e:
            warnings.warn(f"the native host side was not built ({e}): calls take 8 to 13 us of host time instead of 6")
            return None
    binding = sys.modules.get(__package__ + ".binding") if __package__ else None
    if binding is not None:
        binding.load_native()                    # it was imported before there was anything to load
    return host


def build_check(force: bool = False, verbose: bool = False) -> str:
    """The bounds-checked build: every index the verification kernels form is compared with its
    extent and a violation goes to the health word (stand-in for a memory checker; the parity
    tests run a sample of their cases through it)."""
    if force or _stale(LIB_CHECK):
        cmd = [_nvcc(), *NVCC_FLAGS, "-DDD_BOUNDS_CHECK", "-o", LIB_CHECK, *sources()]
        if verbose:
            print(" ".join(cmd), flush=True)
        subprocess.run(cmd, check=True)
    return LIB_CHECK


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose=True,
          extra_flags=["-Xptxas", "-v"] if "--ptxas" in sys.argv else [])
    print(LIB)
    if "--check" in sys.argv:
        print(build_check(force="--force" in sys.argv, verbose=True))
