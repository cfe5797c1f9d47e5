// Device-side building blocks of the Pencil HE hot path on sm_103a:
// 64-bit modular arithmetic (Shoup, Barrett, Harvey lazy butterflies),
// Philox4x64-10, and the parameter structs every kernel receives by value.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

typedef uint64_t u64;
typedef int64_t i64;
typedef uint32_t u32;

#define PENCIL_MAX_LIMBS 4

// ------------------------------------------------------------------ structs
// Per-limb constants for q_j (all computed on the host at context creation).
struct LimbConst {
  u64 q;
  u64 mu;            // floor(2^64 / q)                           (Barrett)
  u64 r64, r64s;     // 2^64 mod q and its Shoup companion
  u64 ninv, ninvs;   // N^{-1} mod q                              (INTT scaling)
  u64 delta, deltas; // floor(q_total / t) mod q                  (BFV Delta)
  uint4 delta_sp;    // its split twiddle (mul_split)
  u64 qtil, qtils;   // (q_total / q_j)^{-1} mod q_j              (CRT)
  u64 th_hi, th_lo;  // floor(2^(128 + t_bits) / q_j), 128 bits   (t / q_j in 0.128 fixed point)
  u64 c60, c64;      // 2^60 mod q and 2^64 mod q                 (split multiply-accumulate folds)
  u64 nqtil, nqtils; // N^{-1} qtil mod q_j                       (INTT scaling folded into the CRT factor)
  u64 a_max;         // floor(2^64 / q) q - 1: the largest 64-bit word accepted for a uniform residue
  // Final scaling kappa of an inverse transform merged into its last stage (split
  // engine): the split twiddles (mul_split) kappa and w1 kappa, w1 = psi^-brv(1) the
  // one twiddle of that stage; kappa = N^{-1} (sc_ninv) or N^{-1} qtil (sc_nqtil).
  uint4 sc_ninv[2];
  uint4 sc_nqtil[2];
  // q = 2^b - cb, sb = b - 32 (mul_split; digits.cuh)
  u64 cb;
  u32 sb;
  u64 digit_bias;    // -(bias of one combination of diagonals) mod q
};

struct DevCtx {
  int log_n;
  int ntt_loge;              // log2(coefficients per thread) of the NTT kernels: 4 or 5
  int n;
  int L;
  int t_bits;
  u64 t_mask;
  LimbConst limb[PENCIL_MAX_LIMBS];
  const ulonglong2* tw_fwd;  // [L][N] (psi^brv(k), Shoup companion)
  const ulonglong2* tw_inv;  // [L][N] (psi^-brv(k), Shoup companion)
  int ntt_arith;             // butterflies of the NTT kernels: 0 Shoup / Harvey, 1 signed split products
  const uint4* tw_fwd_f;     // [L][N] split psi^brv(k) (mul_split)    (null unless every
  const uint4* tw_inv_f;     // [L][N] split psi^-brv(k)                q_j allows them)
  int* status;               // device status word (atomicOr of error bits)
  int mac_split;             // 1: every q_j in (2^59 + 2^33, 2^60) with 2^60, 2^64 mod q_j < 2^28 (30-bit split MAC)
  int mac_nt;                // output columns per thread of the split MAC: 2, 4 or 8
  int mac_staging;           // operand staging of the split MAC: 0 per-thread cp.async ring, 1 bulk copies
  int sms;                   // multiprocessors of the device
  int mac_mma;               // 1: every q_j = 2^b - c with c < 2^(b-32), 2^64 mod q_j < 2^32 (digit products, digits.cuh)
  u64 q_mod_t;               // (q_total mod t): messages are scaled as round(q_total m / t)
  u64 q_frac;                // q_mod_t 2^(64 - t_bits): (q_total mod t) / t as a 64-bit fraction
  int flood_bits;            // 0, or the flooding noise of returned ciphertexts: uniform in [-2^b, 2^b)
};

// A strided view of a user tensor seen as (a, b, r, s) with spatial zero
// padding: element = ptr[base + a*s0 + b*s1 + (r-pr)*s2 + (s-ps)*s3] when
// 0 <= r-pr < hr and 0 <= s-ps < wr, else 0.
struct Accessor {
  const u64* ptr;
  i64 base;
  i64 s0, s1, s2, s3;
  int pr, ps, hr, wr;
};

// Packing of one operand position class (inputs, kernels or outputs) with the strides
// of that operand's tensor: tab[e] = (x) local (a, b, r, s) of coefficient e packed as
// 4 x 16 bits, each below 2^14 (blocks hold at most N <= 2^14 elements), or 0x7fff in
// every field when coefficient e carries nothing, and (y) its offset in bytes from the
// block's first element; org[idx] = the block origin of polynomial idx; bound = the
// geometry extent of (a, b, r, s); support = 1 + the highest e with an entry
// (coefficients from support on are always zero).
struct Packing {
  const ulonglong2* tab;
  const int4* org;
  int4 bound;
  int support;
  const unsigned char* groups;   // [N / 32]: whether any of 32 consecutive coefficients has an entry
  int filled;                    // those groups
  int warps;                     // of the N / 128 runs of 128 coefficients, those with an entry
};

#define PENCIL_TAB_NONE 0x7FFF7FFF7FFF7FFFull

// ------------------------------------------------------------------ 64-bit modular arithmetic
__device__ __forceinline__ u64 mulhi64(u64 a, u64 b) { return __umul64hi(a, b); }

// a * w mod q in [0, 2q), w < q, ws = floor(w 2^64 / q), any a < 2^64 (Shoup).
__device__ __forceinline__ u64 mul_shoup_lazy(u64 a, u64 w, u64 ws, u64 q) {
  u64 qt = mulhi64(a, ws);
  return a * w - qt * q;
}

__device__ __forceinline__ u64 csub(u64 x, u64 q) { return x >= q ? x - q : x; }

__device__ __forceinline__ u64 mul_shoup(u64 a, u64 w, u64 ws, u64 q) {
  return csub(mul_shoup_lazy(a, w, ws, q), q);
}

// x mod q for any x < 2^64 with mu = floor(2^64 / q) (Barrett, one correction).
__device__ __forceinline__ u64 reduce64(u64 x, const LimbConst& c) {
  u64 qt = mulhi64(x, c.mu);
  return csub(x - qt * c.q, c.q);
}

// (hi * 2^64 + lo) mod q, canonical.  Shoup's product accepts any hi < 2^64.
__device__ __forceinline__ u64 reduce128(u64 hi, u64 lo, const LimbConst& c) {
  u64 t = mul_shoup_lazy(hi, c.r64, c.r64s, c.q);  // [0, 2q)
  u64 rl = reduce64(lo, c);
  u64 s = t + rl;                                   // [0, 3q)
  s = csub(s, 2 * c.q);
  return csub(s, c.q);
}

// Alternative formulations measured by pencil_mul_probe (variants 4, 5, 7):
// on GB300 32x32 high products and 32x32->64 products run at half the rate of
// 32-bit multiply-adds, and these variants came out no faster than the
// compiler's Shoup product, so the NTT kernels use Harvey's butterflies below.
//
// a * w mod q in [0, 3q) for ANY a < 2^64, with w < q < 2^62, ws = floor(w 2^64 / q)
// and nq = 2^64 - q.  Shoup's quotient hi64(a * ws) is formed from three
// 32x32->64 multiply-adds (the low x low partial product is dropped, so the
// quotient may be one below Shoup's and the remainder one q above his range
// [0, 2q)); the remainder a * w - qt * q is computed as a * w + qt * nq mod 2^64
// from two more 32x32->64 products and four 32-bit multiply-adds.
__host__ __device__ __forceinline__ u64 mul_shoup3(u64 a, u64 w, u64 ws, u64 nq) {
  const u32 a0 = (u32)a, a1 = (u32)(a >> 32);
  const u32 s0 = (u32)ws, s1 = (u32)(ws >> 32);
  const u64 t = (u64)a0 * s1;
  const u64 u = (u64)a1 * s0 + (u32)t;
  const u64 qt = (u64)a1 * s1 + ((t >> 32) + (u >> 32));
  const u32 w0 = (u32)w, w1 = (u32)(w >> 32);
  const u32 n0 = (u32)nq, n1 = (u32)(nq >> 32);
  const u32 q0 = (u32)qt, q1 = (u32)(qt >> 32);
  const u64 r = (u64)a0 * w0 + (u64)q0 * n0;
  const u32 hi = a1 * w0 + a0 * w1 + q1 * n0 + q0 * n1;
  return r + ((u64)hi << 32);
}

// x - c if x >= c else x, for x < 2^63 and c < 2^63 (sign of the difference).
__host__ __device__ __forceinline__ u64 csub_s(u64 x, u64 c) {
  const u64 d = x - c;
  return ((i64)d < 0) ? x : d;
}

// Cooley-Tukey butterfly on the lazy range [0, 8q) (needs q < 2^60):
// x, y in [0, 8q) -> x + w y, x - w y (mod q) in [0, 8q).
__host__ __device__ __forceinline__ void ct_bf8(u64& x, u64& y, u64 w, u64 ws, u64 nq, u64 q3, u64 q4) {
  const u64 a = csub_s(x, q4);                 // [0, 4q)
  const u64 t = mul_shoup3(y, w, ws, nq);      // [0, 3q)
  x = a + t;                                   // [0, 7q)
  y = a + q3 - t;                              // (0, 7q]
}

// Gentleman-Sande butterfly on the lazy range [0, 4q):
// x, y in [0, 4q) -> x + y, (x - y) w (mod q) in [0, 4q).
__host__ __device__ __forceinline__ void gs_bf4(u64& x, u64& y, u64 w, u64 ws, u64 nq, u64 q4) {
  const u64 s = csub_s(x + y, q4);             // [0, 4q)
  const u64 d = x + q4 - y;                    // (0, 8q)
  x = s;
  y = mul_shoup3(d, w, ws, nq);                // [0, 3q)
}

__device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) { return csub(a + b, q); }

// round((q_total mod t) m / t) for m in [0, t): the part of the BFV message scaling
// round(q_total m / t) = Delta m + this that does not depend on the limb (below t < q_j).
// q_frac m / 2^64 is exact, so rounding adds the top fraction bit.
__device__ __forceinline__ u64 scale_extra(u64 m, const DevCtx& c) {
  return __umul64hi(c.q_frac, m) + ((c.q_frac * m) >> 63);
}
// round(q_total m / t) mod q_j, canonical.
__device__ __forceinline__ u64 scale_msg(u64 m, const LimbConst& lc, const DevCtx& c) {
  return add_mod(mul_shoup(m, lc.delta, lc.deltas, lc.q), scale_extra(m, c), lc.q);
}
__device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) { return a >= b ? a - b : a + q - b; }

// 128-bit accumulate: (hi, lo) += a * b.
__device__ __forceinline__ void mac128(u64& lo, u64& hi, u64 a, u64 b) {
  u64 plo = a * b;
  u64 phi = mulhi64(a, b);
  lo += plo;
  hi += phi + (lo < plo ? 1ull : 0ull);
}

// Harvey Cooley-Tukey butterfly: x, y in [0, 4q) -> x + w y, x - w y in [0, 4q).
__device__ __forceinline__ void ct_butterfly(u64& x, u64& y, u64 w, u64 ws, u64 q, u64 q2) {
  u64 a = x >= q2 ? x - q2 : x;
  u64 t = mul_shoup_lazy(y, w, ws, q);
  x = a + t;
  y = a - t + q2;
}

// Harvey Gentleman-Sande butterfly: x, y in [0, 2q) -> x + y, (x - y) w in [0, 2q).
__device__ __forceinline__ void gs_butterfly(u64& x, u64& y, u64 w, u64 ws, u64 q, u64 q2) {
  u64 s = x + y;
  s = s >= q2 ? s - q2 : s;
  u64 d = x - y + q2;
  x = s;
  y = mul_shoup_lazy(d, w, ws, q);
}

// ------------------------------------------------------------------ pseudo-Mersenne twiddle products
// For q = 2^b - c (c < 2^24 for b = 59, 60, c < 2^(b-33) below; split_prime) and signed lazy
// values y in (-7 2^b, 7.97 2^b).  A twiddle w is kept as its centred representative and that of
// w 2^32 mod q, each split at bit sh = b - 32: w = w1 2^sh + w0 with 0 <= w0 < 2^sh
// and w1 a signed 32-bit word.  With y = y1 2^32 + y0, y0 the SIGNED low word (y1 takes
// its carry), and v the split of w 2^32:
//   H = y0 w1 + y1 v1,  L = y0 w0 + y1 v0     (|H| < 2^63, four signed 32x32->64),
//   y w = L + H 2^sh = L + lo32(H) 2^sh + hi32(H) 2^b = L + lo32(H) 2^sh + hi32(H) c  (mod q):
// the high word of H is the quotient and its low word sits at bit sh, so nothing is
// split by shifts and masks and no quotient is estimated: five wide multiply-adds, two
// shifts, three additions.  The value is signed, for y in [-A, B] (units of 2^b) between
// -(1/2 + A 2^(b-64) + e) and 3/2 + B 2^(b-64) + e with e = max|hi32(H)| c / 2^b <=
// (2^30 + max(A, B) 2^(b-33)) c / 2^b: 1/64 + max(A, B) / 512 for b = 60, twice the first
// term for 59, 1/8 + max(A, B) 2^(b-66) below.  (Shorter primes have the larger e and the
// smaller A and B terms: the ranges of ct_split and gs_split hold for all of them.  Every
// range here is checked in exact fractions, tests/test_split_ranges.py.)  (The unsigned form it replaces
// split w at bit 32 and needed fourteen instructions; measured in registers, a forward
// butterfly with its share of the folds takes 30.0 cycles per warp against 36.7; the low
// word's shift as a sixth wide multiply-add 32.5.)
struct FoldC {
  u32 c, sh, sr, m;   // c, b - 32, 64 - b, 2^(b-32) - 1
  __device__ __forceinline__ explicit FoldC(const LimbConst& lc)
      : c((u32)lc.cb), sh(lc.sb), sr(32u - lc.sb), m((1u << lc.sb) - 1u) {}
};

// base + y w (mod q), lazily.
__device__ __forceinline__ u64 mul_split(u64 base, u64 y, const uint4 w, const FoldC& f) {
  u64 r;
  asm("{\n\t"
      ".reg .u32 y0, y1, s, h0, h1, a, b;\n\t"
      ".reg .u64 l, h, g;\n\t"
      "mov.b64 {y0, y1}, %2;\n\t"
      "shr.u32 s, y0, 31;\n\t"
      "add.u32 y1, y1, s;\n\t"
      "mul.wide.s32 h, y0, %4;\n\t"
      "mad.wide.s32 h, y1, %6, h;\n\t"
      "mad.wide.s32 l, y0, %3, %1;\n\t"
      "mad.wide.s32 l, y1, %5, l;\n\t"
      "mov.b64 {h0, h1}, h;\n\t"
      "mad.wide.s32 l, h1, %7, l;\n\t"
      "shl.b32 a, h0, %8;\n\t"
      "shr.u32 b, h0, %9;\n\t"
      "mov.b64 g, {a, b};\n\t"
      "add.u64 %0, l, g;\n\t"
      "}"
      : "=l"(r)
      : "l"(base), "l"(y), "r"(w.x), "r"(w.y), "r"(w.z), "r"(w.w), "r"(f.c), "r"(f.sh), "r"(f.sr));
  return r;
}

// Signed lazy value, |v| < 2^63 -> (v mod 2^b) + floor(v / 2^b) c, within 2^-7 of [0, 2^b].
__device__ __forceinline__ u64 fold_s(u64 v, const FoldC& f) {
  u64 r;
  asm("{\n\t"
      ".reg .u32 v0, v1, s, h;\n\t.reg .u64 p;\n\t"
      "mov.b64 {v0, v1}, %1;\n\t"
      "shr.s32 s, v1, %3;\n\t"
      "and.b32 h, v1, %4;\n\t"
      "mov.b64 p, {v0, h};\n\t"
      "mad.wide.s32 %0, s, %2, p;\n\t"
      "}"
      : "=l"(r)
      : "l"(v), "r"(f.c), "r"(f.sh), "r"(f.m));
  return r;
}

// The same for an unsigned value below 2^64: below 2^b + 2^(64-b) c < 2 q.
__device__ __forceinline__ u64 fold_u(u64 v, const FoldC& f) {
  u64 r;
  asm("{\n\t"
      ".reg .u32 v0, v1, s, h;\n\t.reg .u64 p;\n\t"
      "mov.b64 {v0, v1}, %1;\n\t"
      "shr.u32 s, v1, %3;\n\t"
      "and.b32 h, v1, %4;\n\t"
      "mov.b64 p, {v0, h};\n\t"
      "mad.wide.u32 %0, s, %2, p;\n\t"
      "}"
      : "=l"(r)
      : "l"(v), "r"(f.c), "r"(f.sh), "r"(f.m));
  return r;
}

// Cooley-Tukey butterfly on signed lazy values: x + w y, x - w y.  From [0, 1] (units
// of 2^b) four stages stay inside (-6.96, 7.96): one fold per round of at most four.
__device__ __forceinline__ void ct_split(u64& x, u64& y, const uint4 w, const FoldC& f) {
  const u64 t = mul_split(0, y, w, f);
  y = x - t;
  x = x + t;
}

// Gentleman-Sande butterfly: x + y, (x - y) w.  From [-0.87, 1.87], two stages with the
// second one's sums folded stay inside (-3.5, 7.5) and return to that range.
__device__ __forceinline__ void gs_split(u64& x, u64& y, const uint4 w, const FoldC& f) {
  const u64 d = x - y;
  x = x + y;
  y = mul_split(0, d, w, f);
}

// [0, 4q) -> [0, q)
__device__ __forceinline__ u64 canon4(u64 x, u64 q, u64 q2) {
  x = x >= q2 ? x - q2 : x;
  return x >= q ? x - q : x;
}

// ------------------------------------------------------------------ Philox4x64-10
// Salmon et al., SC'11: two 64x64->128 products per round on counter words 0
// and 2, high halves mixed with words 1, 3 and the round key; Weyl key schedule.
struct Philox4 {
  u64 v[4];
};

__device__ __forceinline__ Philox4 philox4x64(u64 c0, u64 c1, u64 c2, u64 c3, u64 k0, u64 k1) {
  const u64 M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
  const u64 W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += W0;
      k1 += W1;
    }
    u64 lo0 = M0 * c0, hi0 = mulhi64(M0, c0);
    u64 lo1 = M1 * c2, hi1 = mulhi64(M1, c2);
    u64 n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
  Philox4 o;
  o.v[0] = c0;
  o.v[1] = c1;
  o.v[2] = c2;
  o.v[3] = c3;
  return o;
}

// Stream domains (the second key word).
#define PENCIL_DOM_SECRET 1ull
#define PENCIL_DOM_A 2ull
#define PENCIL_DOM_E 3ull
#define PENCIL_DOM_MASK 4ull
#define PENCIL_DOM_MASK_PAD 5ull
#define PENCIL_DOM_FLOOD 6ull
#define PENCIL_DOM_PK_A 7ull    // public key's a
#define PENCIL_DOM_PK_E 8ull    // public key's error
#define PENCIL_DOM_PK_U 9ull    // public-key encryption's ternary u
#define PENCIL_DOM_PK_E2 10ull  // public-key encryption's e2 (its e1 is PENCIL_DOM_E)

__device__ __forceinline__ u64 philox_word(const Philox4& w, int i) {
  return i == 0 ? w.v[0] : i == 1 ? w.v[1] : i == 2 ? w.v[2] : w.v[3];
}

// 64-bit word of coefficient `coef` whose residue mod q_j is uniform (the encryption
// mask a, the public key's a), from its Philox word w: w is accepted when w <= a_max
// (below the largest multiple of q_j under 2^64); a rejected word is replaced by word 0
// of the block at counter (coef, ct, limb, r), r = 1, 2, ... (probability below 2^-32
// per word for the primes used; the loop stops after 64 replacements, which for primes
// above 2^40 never happens in practice).
__device__ __forceinline__ u64 uniform_word(u64 w, int coef, int ct, int limb, u64 seed, u64 dom,
                                            const LimbConst& lc) {
  for (u64 r = 1; w > lc.a_max && r <= 64; ++r) w = philox4x64((u64)coef, (u64)ct, (u64)limb, r, seed, dom).v[0];
  return w;
}

// ------------------------------------------------------------------ packing gathers
// One polynomial's view of its operand: address of its block's first element (or, with
// a null tensor, that element's index times 8) and the extent of its valid local
// coordinates, packed so that one 64-bit subtraction tests all four upper bounds and one
// 32-bit addition the two lower ones: with 16-bit fields c <= 0x7fff, bit 15 of
// (0x8000 + max) - c is set iff c <= max and bit 15 of c + (0x8000 - min) iff c >= min.
// Set up once per polynomial; an element then costs a 16-byte table load, six integer
// operations and a 64-bit addition (the origin, four compares, two range checks and four
// 64-bit strided products it replaces were about half of the fused transforms'
// prologues: ModeMoPrep at N = 8192 260 thread instructions per coefficient, 175 of them
// the transform).
struct Window {
  const char* base;
  u32 tl, th, lh;
  __device__ __forceinline__ Window(const Packing& pk, const Accessor& ac, int idx, const void* ptr) {
    const int4 o = __ldg(pk.org + idx);
    base = reinterpret_cast<const char*>(ptr) +
           8 * (ac.base + o.x * ac.s0 + o.y * ac.s1 + (i64)(o.z - ac.pr) * ac.s2 + (i64)(o.w - ac.ps) * ac.s3);
    tl = top(pk.bound.x - o.x) | (top(pk.bound.y - o.y) << 16);
    th = top(min(pk.bound.z, ac.hr + ac.pr) - o.z) | (top(min(pk.bound.w, ac.wr + ac.ps) - o.w) << 16);
    lh = low(ac.pr - o.z) | (low(ac.ps - o.w) << 16);
  }
  __device__ __forceinline__ Window(const char* b, u32 l, u32 h, u32 m) : base(b), tl(l), th(h), lh(m) {}
  static __device__ __forceinline__ u32 top(int extent) { return 0x7FFFu + (u32)min(max(extent, 0), 0x4000); }
  static __device__ __forceinline__ u32 low(int first) { return 0x8000u - (u32)min(max(first, 0), 0x7FFF); }
  __device__ __forceinline__ bool has(const ulonglong2& ent) const {
    const u32 cl = (u32)ent.x, ch = (u32)(ent.x >> 32);
    return ((tl - cl) & (th - ch) & (ch + lh) & 0x80008000u) == 0x80008000u;
  }
  __device__ __forceinline__ const char* at(const ulonglong2& ent) const { return base + (i64)ent.y; }
  // element of coefficient e (0 where the coefficient carries nothing)
  __device__ __forceinline__ u64 get(const Packing& pk, int e) const {
    const ulonglong2 ent = __ldg(pk.tab + e);
    return has(ent) ? __ldg(reinterpret_cast<const u64*>(at(ent))) : 0ull;
  }
  // element index of coefficient e in the operand's tensor (null ptr), or -1
  __device__ __forceinline__ i64 index(const ulonglong2& ent) const { return has(ent) ? (i64)at(ent) >> 3 : -1; }
  __device__ __forceinline__ i64 index(const Packing& pk, int e) const { return index(__ldg(pk.tab + e)); }
};

// Decryption's CRT step: with y_j = x_j (q/q_j)^{-1} mod q_j,
//   t x / q = sum_j y_j t / q_j - v t  (v integer),
// so round(t x / q) mod t = round(sum_j y_j th_j / 2^128) mod t with
// th_j = floor(2^(128 + t_bits) / q_j).  The sum is kept as a 128-bit window
// (64 integer bits, 64 fraction bits); truncation error < L * 2^-63.
struct CrtSum {
  u64 lo, hi;
};
__device__ __forceinline__ void crt_add(CrtSum& s, u64 y, const LimbConst& lc) {
  const u64 a_hi = __umul64hi(y, lc.th_lo);
  const u64 b_lo = y * lc.th_hi;
  const u64 b_hi = __umul64hi(y, lc.th_hi);
  const u64 w_lo = b_lo + a_hi;
  const u64 w_hi = b_hi + (w_lo < b_lo ? 1ull : 0ull);
  s.lo += w_lo;
  s.hi += w_hi + (s.lo < w_lo ? 1ull : 0ull);
}
// The rounded value mod t; with `check`, flags (status bit 0) a fraction within
// 1/4 of one half (noise too close to the decryption bound).
__device__ __forceinline__ u64 crt_round(const CrtSum& s, u64 t_mask, int check, int* status) {
  if (check) {
    const i64 frac = (i64)s.lo;   // signed distance to the nearest integer, units of 2^-64
    const u64 mag = frac < 0 ? (u64)(-frac) : (u64)frac;
    if (mag >= (1ull << 62)) atomicOr(status, 1);
  }
  const u64 r_lo = s.lo + (1ull << 63);
  const u64 r_hi = s.hi + (r_lo < s.lo ? 1ull : 0ull);
  return r_hi & t_mask;
}
