"""csrc/rules.h compiled for the host: the rules that split and choose launches, as the
library uses them, without a GPU."""
import ctypes
import functools
import os
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2403_11166_gb300", "csrc")
SHIM = r"""
#include "rules.h"
using namespace pencil;
extern "C" void ring_split_(long long K, long long tiles, int sms, int* out) {
  const RingSplit r = ring_split(K, tiles, sms);
  out[0] = r.chunks;
  out[1] = r.per;
  out[2] = r.parts;
}
extern "C" long long ring_launch_k() { return kRingLaunchK; }
"""


@functools.lru_cache(maxsize=None)
def load() -> ctypes.CDLL:
    d = tempfile.mkdtemp()
    src, out = os.path.join(d, "rules.cpp"), os.path.join(d, "rules.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-fsanitize=undefined",
                    "-fno-sanitize-recover=all", "-I", CSRC, src, "-o", out], check=True)
    return ctypes.CDLL(out)


def ring_split(k: int, tiles: int, sms: int = 152):
    """(chunks, chunks of a part, parts) of one launch"""
    out = (ctypes.c_int * 3)()
    load().ring_split_(ctypes.c_longlong(k), ctypes.c_longlong(tiles), sms, out)
    return tuple(out)


def ring_launch_k() -> int:
    load().ring_launch_k.restype = ctypes.c_longlong
    return load().ring_launch_k()
