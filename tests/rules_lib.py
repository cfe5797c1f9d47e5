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
extern "C" int ring_form_(long long outs, const int* d, int wide, int sms) {
  return (int)ring_form(RingShape{outs, d[0], d[1], d[2], d[3], d[4], d[5], wide != 0}, sms);
}
extern "C" int bias_parts_(long long elements) { return bias_parts(elements); }
extern "C" int lincomb_pairs_(long long count) { return lincomb_pairs(count); }
extern "C" int split_prime_(unsigned long long q) { return split_prime(q); }
extern "C" void split_words_(unsigned long long w, unsigned long long q, unsigned* out) {
  const SplitWords s = split_words(w, q);
  for (int i = 0; i < 4; ++i) out[i] = s.v[i];
}
extern "C" int mac_form_(int digits, int split, int columns, int staging, int rows, int K, int NC, int dual) {
  return (int)mac_form(MacKnobs{digits != 0, split != 0, columns, staging}, rows, K, NC, dual != 0);
}
extern "C" int mask_skips_(long long count, int n, int warps, int sms) { return mask_skips(count, n, warps, sms); }
extern "C" int compact_skips_(int n, int filled) { return compact_skips(n, filled); }
"""
MAC_FORMS = ("generic", "smem", "ring", "bulk", "short", "digits")
RING_FORMS = ("tile", "offsets", "outputs", "digits")


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


def ring_form(layer, role: int, t_bits: int, sms: int = 152) -> str:
    """Form of a plaintext correlation; layer = (B, Ci, Co, H, kernel, pad), fully connected
    ones with H = kernel = 1; role 0 forward, 1 input gradient, 2 weight gradient."""
    b, ci, co, h, k, pad = layer
    ho = h + 2 * pad - k + 1
    if role == 0:
        outs, dims = b * co * ho * ho, (co, ci, k, k, ho, ho)
    elif role == 1:
        outs, dims = b * ci * h * h, (ci, co, k, k, h, h)
    else:
        outs, dims = ci * co * k * k, (co, b, ho, ho, k, k)
    return RING_FORMS[load().ring_form_(ctypes.c_longlong(outs), (ctypes.c_int * 6)(*dims), int(t_bits > 48), sms)]


def lincomb_pairs(count: int) -> bool:
    return bool(load().lincomb_pairs_(ctypes.c_longlong(count)))


def split_prime(q: int) -> bool:
    return bool(load().split_prime_(ctypes.c_ulonglong(q)))


def split_words(w: int, q: int):
    """(low, rest) of w and of w 2^32 mod q, the rests signed."""
    out = (ctypes.c_uint * 4)()
    load().split_words_(ctypes.c_ulonglong(w), ctypes.c_ulonglong(q), out)
    signed = [v - (1 << 32) if v >> 31 else v for v in out]
    return (out[0], signed[1]), (out[2], signed[3])


def mac_form(rows: int, k: int, nc: int, dual: bool = False, split: bool = True, columns: int = 4, staging: int = 1) -> str:
    """Form of a single multiply-accumulate; split: the context's primes are the 60-bit ones
    (else other primes that digit products take)."""
    return MAC_FORMS[load().mac_form_(1, int(split), columns, staging, rows, k, nc, int(dual))]


def mask_skips(count: int, n: int, warps: int, sms: int = 152) -> bool:
    return bool(load().mask_skips_(ctypes.c_longlong(count), n, warps, sms))
