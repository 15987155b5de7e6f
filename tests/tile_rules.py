"""The launchers' tile arithmetic (csrc/tile_rules.h), compiled for the host."""
import ctypes
import functools
import os
import subprocess
import tempfile

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_04985_b200", "csrc")

SOURCE = """
#include "tile_rules.h"
extern "C" int mma_width(int n) { return fpt::umma_i8_pair_width(n); }
extern "C" int pair_width(int M, int N, int pairs) { return fpt::pair_tile_width(M, N, pairs); }
"""


@functools.lru_cache(None)
def rules():
    with tempfile.TemporaryDirectory() as tmp:
        src, lib = os.path.join(tmp, "rules.cpp"), os.path.join(tmp, "librules.so")
        with open(src, "w") as f:
            f.write(SOURCE)
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib], check=True)
        return ctypes.CDLL(lib)
