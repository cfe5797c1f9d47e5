// Host-side rules that split and choose launches by sizes, in plain C++ (no CUDA types),
// so that they can be compiled and checked without a GPU.
#pragma once
#include <algorithm>

namespace pencil {

// ------------------------------------------------------------------ split products
inline int bit_length(unsigned long long q) { return 64 - __builtin_clzll(q); }

// Whether mul_split (common.cuh) takes the prime q = 2^b - c: c < 2^24 for b = 59, 60 and
// c < 2^(b-33) below; b >= 40.
inline bool split_prime(unsigned long long q) {
  const int b = bit_length(q);
  if (b < 40 || b > 60) return false;
  return (1ull << b) - q < (b >= 59 ? 1ull << 24 : 1ull << (b - 33));
}

// Split twiddle of mul_split for a split_prime q of b bits: the centred representatives of
// w < q and of w 2^32 mod q, each as (low b - 32 bits, signed rest).
struct SplitWords {
  unsigned v[4];
};
inline SplitWords split_words(unsigned long long w, unsigned long long q) {
  const int sh = bit_length(q) - 32;
  const unsigned long long v[2] = {w, (unsigned long long)(((unsigned __int128)w << 32) % q)};
  SplitWords out;
  for (int i = 0; i < 2; ++i) {
    const long long x = v[i] > q / 2 ? (long long)(v[i] - q) : (long long)v[i];
    out.v[2 * i] = (unsigned)((unsigned long long)x & ((1ull << sh) - 1));
    out.v[2 * i + 1] = (unsigned)(int)(x >> sh);
  }
  return out;
}

// ------------------------------------------------------------------ multiply-accumulate
// What a context allows and asks for (DevCtx: mac_mma, mac_split, mac_nt, mac_staging).
struct MacKnobs {
  bool digits, split;
  int columns, staging;
};

enum class MacForm {
  kGeneric,   // k_mac: any prime
  kSmem,      // k_mac_smem: columns 0
  kRing,      // k_mac_ring: staging 0
  kBulk,      // k_mac_bulk
  kShort,     // k_mac_short: Alg. 1 with at most kMacShortK input blocks
  kDigits     // k_mac_mma: digit products on the tensor cores
};
constexpr int kMacShortK = 6;

// Digit products on the tensor cores (mac_mma.cu) against the integer multiply-add
// kernels, by modelled time of one slot's block in common units.  A tensor-core tile
// is 16 columns n x 4 rows m (Alg. 2: 8 rows of one component) whatever part of it
// exists and pays its combination once per chunk of 16 (8) input blocks; the integer
// kernels pay per existing (m, n) pair and input block.  Fitted to launches on GB300
// at L N = 24576 (us; tensor cores / k_mac_bulk): M = 30, NC = 64: K = 3 605 / 510,
// 5 657 / 651, 6 657 / 768, 16 875 / 1542, 32 1582 / 2871; M = 10, NC = 16: K = 6
// 74 / 72, 8 75 / 84, 16 91 / 138; M = 4, NC = 4: K = 16 36 / 25, 32 65 / 42; M = 2,
// NC = 64: K = 16 150 / 114.  Two 54-bit primes at N = 4096 (k_mac): M = 10, NC = 16:
// K = 1 24 / 22, 2 24 / 28, 16 38 / 129.  (Single launches with split-form primes take
// k_mac_short up to K = 6; there the rule decides for the batch engine's items only.)
inline bool mac_digits_win(const MacKnobs& c, int rows, int K, int NC, bool dual) {
  if (!c.digits || c.columns == 0 || c.staging != 1) return false;   // not available, or tuned away
  const double k = K, nt = (NC + 15) / 16, pairs = (double)rows * NC / 64.0;
  if (dual) return 2.0 * ((rows + 7) / 8) * nt * 22.0 * ((K + 7) / 8) < pairs * (c.split ? 11.0 + 6.0 * k : 15.0 + 13.0 * k);
  const double unit = K <= 16 ? 19.0 + 0.7 * k : 26.0 * ((K + 15) / 16);
  return ((rows + 3) / 4) * nt * unit < pairs * (c.split ? 11.0 + 2.65 * k : 15.0 + 6.6 * k);
}

// Form of a single launch of output rows x NC products over K input blocks.
inline MacForm mac_form(const MacKnobs& c, int rows, int K, int NC, bool dual) {
  if (!dual && c.split && c.columns != 0 && c.staging == 1 && K >= 1 && K <= kMacShortK)
    return MacForm::kShort;   // faster than both at every size measured
  if (mac_digits_win(c, rows, K, NC, dual)) return MacForm::kDigits;
  if (!c.split) return MacForm::kGeneric;
  return c.columns == 0 ? MacForm::kSmem : c.staging == 1 ? MacForm::kBulk : MacForm::kRing;
}

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


// Sizes of one correlation (kernels.h, RingParams): `wide` = t > 2^48 (eight digits, not six).
struct RingShape {
  long long outs;
  int Co, Ci, KH, KW, Ho, Wo;
  bool wide;
  long long positions() const { return outs / Co; }
  long long K() const { return (long long)Ci * KH * KW; }
};

enum class RingForm {
  kTile,      // k_ring_tile: a thread = 4 positions x 4 or 8 channels, the whole reduction
  kOffsets,   // k_ring_wgrad: a CTA = all kernel offsets of one (a, o)
  kOutputs,   // k_ring_block: a CTA = one output
  kDigits     // k_ring_mma: digit products on the tensor cores
};

// Output tile of the tensor-core form: rows (channels), columns (positions), CTAs per SM.
struct RingTile {
  int rows, cols, per_sm;
};
inline RingTile ring_tile(int Co) {
  return Co > 32 ? RingTile{64, 64, 2} : Co > 16 ? RingTile{32, 64, 3} : RingTile{16, 128, 3};
}

// Modelled times of the forms, us.  Fitted to 3174 sizes on GB300 (positions 1 .. 200704,
// reductions of 1 .. 100 000, 1 .. 1000 channels, t = 2^41 and 2^59): tensor cores within 7 %
// (rms), tile 10 %, offsets 14 %, outputs 8 %; choosing by them costs 0.2 % over the faster
// of the forms' measured times (geometric mean).
inline double ring_digits_us(const RingShape& s, int sms) {
  const RingTile t = ring_tile(s.Co);
  const long long tiles = ((s.positions() + t.cols - 1) / t.cols) * ((s.Co + t.rows - 1) / t.rows);
  const RingSplit p = ring_split(s.K(), tiles, sms);   // (a longer reduction's first launch)
  // waves of CTAs; a chunk takes a full SM 2.75 us (rows 64: 3.05), a lone CTA 1.6
  const long long ctas = tiles * p.parts, cap = (long long)t.per_sm * sms, rest = ctas % cap;
  const double full = t.rows == 64 ? 3.05 : 2.75;
  const double wave = (double)(ctas / cap) * full + (rest ? std::max(1.6, full * (double)rest / (double)cap) : 0.0);
  return 0.3 + 2.75 * std::min(1.0, (double)s.positions() / 64) + (t.rows == 64 ? 1.7 : 0.0) +
         (p.parts > 1 ? 2.9 : 0.0) + wave * (p.per * (s.wide ? 1.28 : 1.0) + 1.5);
}

// a serial part (latency of one thread's loop) and a parallel one (work over the GPU)
inline double ring_overlap_us(double serial, double work, double share) {
  return std::max(serial, work) + share * std::min(serial, work);
}

inline double ring_tile_us(const RingShape& s) {
  const int ot = s.Co >= 8 ? 8 : 4;
  const double K = (double)s.K(), lines = K / s.KW, groups = (s.Co + ot - 1) / ot;
  return 2.0 + 1.5 * std::min(1.0, (double)s.positions() / 8) +
         ring_overlap_us((0.36 * K + 0.185 * lines) * (ot == 8 ? 1.42 : 1.0),
                         (double)s.positions() * groups * (0.247 * ot * K + 1.55 * lines + 3.9 * std::min(ot, s.Co)) * 1e-6,
                         0.64);
}

inline double ring_offsets_us(const RingShape& s) {
  const double h = (double)s.Ho * s.Wo, steps = (double)s.Ci * (((long long)s.KH * s.KW + 255) / 256);
  return 1.94 + ring_overlap_us(steps * (0.205 + 0.049 * h),
                                (double)s.outs / h * (steps * (0.158 * h + 0.41) + 0.33 * h) * 1e-3, 0.37);
}

inline double ring_outputs_us(const RingShape& s) {
  const double steps = (double)s.Ci * (((long long)s.KH * s.KW + 255) / 256);
  return 2.17 + ring_overlap_us(0.317 * steps, (double)s.outs * (steps + 2.8) * 0.59e-3, 0.61);
}

// The tensor cores take a correlation unless its integer form is faster: short reductions
// (a chunk of 16 is paid whole), weight gradients of few images (the split's two extra
// passes), few channels over many positions (at most 4 of a tile's 16 rows exist), above
// all with t > 2^48.  Integer form by the kernel's elements: 256 or more (weight gradients)
// share them over a CTA's threads.  Measured (us, integer / tensor cores): fc 64 x 2048 to 2
// weights, batch 1, K = 1 4.9 / 9.5; 28 x 28 image's 3 x 3 weight gradient, 3 to 64 channels,
// batch 1 4.8 / 17.5, batch 8 41 / 14; conv3x3 64->3, 56x56, batch 64 379 / 374 (t = 2^41),
// 381 / 468 (t = 2^59); fc 2048 to 2, batch 64 1240 / 13 (t = 2^59: / 14.5).
inline RingForm ring_form(const RingShape& s, int sms) {
  const bool cta = (long long)s.KH * s.KW >= 256 && s.outs < 1ll << 31;
  const bool offsets = cta && s.Ho == s.Wo && (s.Ho == 1 || s.Ho == 3 || s.Ho == 5);
  const RingForm integer = offsets ? RingForm::kOffsets : cta ? RingForm::kOutputs : RingForm::kTile;
  const double us = offsets ? ring_offsets_us(s) : cta ? ring_outputs_us(s) : ring_tile_us(s);
  return us < ring_digits_us(s, sms) ? integer : RingForm::kDigits;
}

// CTAs (one cluster) per channel of a bias gradient over `elements` each: one takes 16
// elements a thread; a cluster's launch costs as much.
inline int bias_parts(long long elements) { return elements > 4096 ? 8 : 1; }

// Whether a linear combination's threads take two elements each (where everything is
// aligned for it): below, twice the threads hide more latency (us, one / two: 65536 elements
// of 64 terms 5.2 / 5.7, of 4 2.2 / 2.2; 150 000 6.8 / 6.7 and 2.5 / 2.4; 2^20 81.2 / 80.3 and
// 6.6 / 5.1).
inline bool lincomb_pairs(long long count) { return count >= 1 << 17; }

// Whether `count` mask polynomials, of whose n / 128 runs of 128 coefficients `warps` carry
// outputs, are drawn by the form that skips the others (k_mask_poly): a fifth of them or more
// are empty and the launch has two CTAs of 1024 coefficients for every SM (a smaller one is
// one CTA's latency, which the test lengthens: 2 polynomials 3.6 / 3.9 us).
inline bool mask_skips(long long count, int n, int warps, int sms) {
  return 5ll * (n / 128 - warps) >= n / 128 && count * (n / 1024) >= 2ll * sms;
}

// Whether the compact form of polynomials, of whose n / 32 groups of 32 coefficients `filled`
// carry outputs, is stored by the epilogue that skips the others (ModeCompactFew): half of
// them are empty (us, all looked up / skipping: 2048 polynomials at N = 8192 with 31 % 460 /
// 408, 2752 with 5 % 606 / 497, 1920 with 98 % 444 / 461).
inline bool compact_skips(int n, int filled) { return 2 * filled <= n / 32; }

}  // namespace pencil
