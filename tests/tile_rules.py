"""The launchers' tile arithmetic (csrc/tile_rules.h), compiled for the host."""
import collections
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
extern "C" int ahead(int M, int N, int K, int pairs, int extras, int swiglu) {
  return swiglu ? fpt::wt_ahead_swiglu(M, N, K, pairs) : fpt::wt_ahead(M, N, K, pairs, extras);
}
extern "C" void cut(int M, int N, int K, int pairs, int quads, long long* out) {
  const fpt::WtCut c = fpt::wt_cut(M, N, K, pairs, quads);
  out[0] = c.tn; out[1] = c.ksplit; out[2] = c.ns;
}
"""
Cut = collections.namedtuple("Cut", "tokens shared ns tiles")


@functools.lru_cache(None)
def rules():
    with tempfile.TemporaryDirectory() as tmp:
        src, lib = os.path.join(tmp, "rules.cpp"), os.path.join(tmp, "librules.so")
        with open(src, "w") as f:
            f.write(SOURCE)
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib], check=True)
        return ctypes.CDLL(lib)


def wt_ahead(M, N, K, extras=0, swiglu=False, pairs=74):
    """Whether a linear (swiglu: the gate||up matmul of a block of more than 128 tokens) takes the kernel for one-byte codes."""
    return bool(rules().ahead(M, N, K, pairs, extras, int(swiglu)))


def wt_cut(M, N, K, pairs=74, quads=33):
    """How the kernel for one-byte codes cuts M tokens x N outputs x K (74 CTA pairs and 33 clusters of four fit a B200)."""
    out = (ctypes.c_longlong * 3)()
    rules().cut(M, N, K, pairs, quads, out)
    return Cut(out[0], out[1] == 2, out[2], -(-M // out[0]) * -(-N // 256))
