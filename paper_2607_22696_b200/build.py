"""Compile the 3D-DSA CUDA library for sm_100a into libdsa3d.so next to this file."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libdsa3d.so")
LIB_AUTOGRAD = os.path.join(HERE, "_autograd_native.so")  # the torch.autograd functions, linked against LIB
LIB_DEBUG = os.path.join(HERE, "libdsa3d_debug.so")     # the checked build (-DDSA3D_DEBUG)
SOURCES = ["dsa3d_api.cu", "dsa3d_forward.cu", "dsa3d_backward.cu", "dsa3d_cells.cu", "dsa3d_noalloc.cu", "dsa3d_probes.cu",
           "dsa3d_producer.cu", "dsa3d_fixed_window.cu", "dsa3d_fixed_window_planes.cu", "dsa3d_fixed_window_tables.cu",
           "dsa3d_fixed_window_backward.cu", "dsa3d_fixed_window_tile_grad.cu",
           "dsa3d_fixed_window_planes_grad.cu", "dsa3d_bounded_offsets_backward.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-lineinfo", "-std=c++17",
              "-Xcompiler", "-fPIC"]


def _nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    built = os.path.getmtime(lib)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + \
           [os.path.join(os.path.dirname(HERE), "include", "dsa3d.h")]
    return any(os.path.getmtime(p) > built for p in deps)


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Build libdsa3d.so (or, with debug=True, the bounds-checked libdsa3d_debug.so) if it is missing
    or older than its sources; return its path."""
    lib = LIB_DEBUG if debug else LIB
    if not debug:
        _compile(lib, force, verbose, debug)
        build_autograd(force)
        return lib
    return _compile(lib, force, verbose, debug)


def build_autograd(force: bool = False) -> str:
    """Build the compiled torch.autograd functions (against torch's own headers); return the path."""
    if not force and not _stale(LIB_AUTOGRAD):
        return LIB_AUTOGRAD
    import sysconfig

    import torch
    top = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(_nvcc())) or "/usr/local/cuda"
    include = [os.path.join(top, "include"), os.path.join(top, "include", "torch", "csrc", "api", "include"),
               os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    cmd = ["g++", "-shared", "-fPIC", "-O2", "-std=c++17", "-o", LIB_AUTOGRAD, os.path.join(CSRC, "dsa3d_autograd.cpp"),
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-DTORCH_EXTENSION_NAME=_autograd_native"]
    cmd += [f"-I{p}" for p in include]
    cmd += [f"-L{os.path.join(top, 'lib')}", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch", "-ltorch_python",
            f"-L{HERE}", "-l:" + os.path.basename(LIB), "-Wl,-rpath,$ORIGIN"]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError("g++ failed:\n" + res.stdout + res.stderr)
    return LIB_AUTOGRAD


def _compile(lib: str, force: bool, verbose: bool, debug: bool) -> str:
    if not force and not _stale(lib):
        return lib
    flags = list(NVCC_FLAGS) + os.environ.get("DSA3D_NVCC_EXTRA", "").split() + (["-DDSA3D_DEBUG"] if debug else [])
    if verbose:
        flags += ["-Xptxas", "-v"]
    cmd = [_nvcc(), "-t", "0", "-shared", "-o", lib] + flags + [os.path.join(CSRC, s) for s in SOURCES]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    return lib


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv))
