"""Small host programs over the library's own planning code (csrc/swin_kernels.h), for tests that need no GPU."""
import os
import subprocess

from paper_2608_15211_b200.build import CSRC, build

PRELUDE = """
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include "terra.h"
#include "swin_kernels.h"
#include "win_tiles.cuh"
namespace terra { int resolve_attention_geo(const terra_swin_desc* d, Geo* out); }
using namespace terra;
"""


def run_host_program(tmp_path, source, *args):
    """Compiles `source` behind the prelude, links it with the built library and runs it; its output, or AssertionError."""
    lib = build()
    src, exe = str(tmp_path / "program.cu"), str(tmp_path / "program")
    with open(src, "w") as f:
        f.write(PRELUDE + source)
    nvcc = os.environ.get("NVCC", "nvcc")
    include = os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include")
    proc = subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_100a,code=sm_100a", "-I" + CSRC, "-I" + include, "-o", exe, src, lib,
                           "-Xlinker", "-rpath," + os.path.dirname(lib)], capture_output=True, text=True)
    assert proc.returncode == 0, proc.stdout + proc.stderr
    proc = subprocess.run([exe, *map(str, args)], capture_output=True, text=True)
    assert proc.returncode == 0, proc.stdout[-4000:] + proc.stderr[-4000:]
    return proc.stdout
