"""Builds the CUDA library in-tree for sm_100a with nvcc (cross-compiles without a GPU), and the binding's native module."""
from __future__ import annotations

import glob
import importlib.metadata
import os
import subprocess
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libterra_swin.so")
HOST_SRC = os.path.join(CSRC, "host_module.cpp")
HOST_PATH = os.path.join(PKG_DIR, "_host.so")
HOST_TAG_PATH = HOST_PATH + ".tag"          # the Python and torch that the native module was built for

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--shared", "-Xcompiler", "-fPIC", "-lcuda"]


def sources() -> list[str]:
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    built = os.path.getmtime(LIB_PATH)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(os.path.dirname(PKG_DIR), "include", "*.h"))
    return any(os.path.getmtime(p) > built for p in deps)


def _host_tag() -> str:
    return f"{sysconfig.get_config_var('SOABI')} torch {importlib.metadata.version('torch')}"


def _host_stale() -> bool:
    if not os.path.exists(HOST_PATH) or not os.path.exists(HOST_TAG_PATH):
        return True
    header = os.path.join(os.path.dirname(PKG_DIR), "include", "terra.h")
    if os.path.getmtime(HOST_PATH) < max(os.path.getmtime(HOST_SRC), os.path.getmtime(header)):
        return True
    with open(HOST_TAG_PATH) as f:
        return f.read() != _host_tag()


def build_host(force: bool = False) -> str:
    """Compile csrc/host_module.cpp, the attention calls' argument handling, against the installed Python and torch."""
    if not force and not _host_stale():
        return HOST_PATH
    import torch
    from torch.utils import cpp_extension
    lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = cpp_extension.CUDA_HOME or "/usr/local/cuda"
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-o", HOST_PATH, HOST_SRC]
    cmd += ["-I" + d for d in cpp_extension.include_paths() + [sysconfig.get_paths()["include"], os.path.join(cuda, "include")]]
    cmd += ["-L" + lib, "-Wl,-rpath," + lib, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-ltorch_cuda", "-lc10", "-lc10_cuda"]
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if proc.returncode != 0:
        raise RuntimeError("g++ failed:\n" + proc.stdout + proc.stderr)
    with open(HOST_TAG_PATH, "w") as f:
        f.write(_host_tag())
    return HOST_PATH


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libterra_swin.so and the native module next to this file; returns the library's path."""
    build_host(force)
    if not force and not _stale():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB_PATH] + sources()
    proc = subprocess.run(cmd, capture_output=True, text=True)
    if proc.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + proc.stdout + proc.stderr)
    if verbose:
        print(proc.stderr)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force=True, verbose=True))
