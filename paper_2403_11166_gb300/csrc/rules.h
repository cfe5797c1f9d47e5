// Host-side rules that split and choose launches by sizes, in plain C++ (no CUDA types),
// so that they can be compiled and checked without a GPU.
#pragma once
#include <algorithm>

namespace pencil {

// ------------------------------------------------------------------ plaintext correlations
// Reduction of one tensor-core launch in parts of whole 16-element chunks.
struct RingSplit {
  int chunks;   // chunks of 16
  int per;      // chunks of one part
  int parts;    // parts > 1 add with atomics
};

// Elements of a reduction that one launch takes (chunk numbers fit 32 bits); a longer one
// (an operand of more than 64 GiB) takes several launches.
constexpr long long kRingLaunchK = 1ll << 33;

// `tiles` output tiles on `sms` multiprocessors, K <= kRingLaunchK: up to three CTAs per SM,
// at least four chunks in a part.
inline RingSplit ring_split(long long K, long long tiles, int sms) {
  RingSplit r;
  r.chunks = (int)((std::min(K, kRingLaunchK) + 15) / 16);
  long long parts = std::max<long long>(1, 3ll * sms / std::max<long long>(1, tiles));
  parts = std::min<long long>(parts, std::max(1, r.chunks / 4));
  r.per = (int)((r.chunks + parts - 1) / parts);
  r.parts = (r.chunks + r.per - 1) / r.per;
  return r;
}

}  // namespace pencil
