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
extern "C" int ring_split_(long long K, long long tiles, int sms, unsigned* out) {
  RingSplit r;
  if (!ring_split(K, tiles, sms, &r)) return 0;
  out[0] = r.chunks;
  out[1] = r.per;
  out[2] = r.parts;
  return 1;
}
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
    """(chunks, chunks of a part, parts), or None where the length is refused."""
    out = (ctypes.c_uint * 3)()
    ok = load().ring_split_(ctypes.c_longlong(k), ctypes.c_longlong(tiles), sms, out)
    return tuple(out) if ok else None
