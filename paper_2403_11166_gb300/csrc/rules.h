// Host-side rules that split and choose launches by sizes, in plain C++ (no CUDA types),
// so that they can be compiled and checked without a GPU.
#pragma once
#include <algorithm>

namespace pencil {

// ------------------------------------------------------------------ plaintext correlations
// Reduction of the tensor-core form in parts of whole 16-element chunks.
struct RingSplit {
  unsigned chunks;   // chunks of 16
  unsigned per;      // chunks of one part
  unsigned parts;    // parts > 1 add with atomics
};

// `tiles` output tiles on `sms` multiprocessors: up to three CTAs per SM, at least four
// chunks in a part.  False for a reduction of 3 2^34 elements or more (an operand of at
// least 384 GiB): below, chunk numbers and their next three fit 32 bits unsigned.
inline bool ring_split(long long K, long long tiles, int sms, RingSplit* r) {
  if (K < 1 || K >= 3ll << 34) return false;
  r->chunks = (unsigned)((K + 15) / 16);
  long long parts = std::max<long long>(1, 3ll * sms / std::max<long long>(1, tiles));
  parts = std::min<long long>(parts, std::max(1u, r->chunks / 4));
  r->per = (unsigned)((r->chunks + parts - 1) / parts);
  r->parts = (unsigned)((r->chunks + (long long)r->per - 1) / r->per);
  return true;
}

}  // namespace pencil
