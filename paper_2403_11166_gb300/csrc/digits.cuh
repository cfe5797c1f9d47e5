// Exact integer contractions on the tensor cores.
//
// A 64-bit word is eight base-256 digits.  A digit b (0 .. 255) placed in the low
// byte of an f16 is the subnormal b 2^-24, exactly; products of two digits are
// multiples of 2^-48 and an f32 accumulator that starts at 2^-25 has that unit in
// its last place, so after any sum n < 2^23 of digit products its bit pattern is
// kDigitBias + n: no conversion on the way in or out.  Diagonal d of a product
// holds sum_k sum_{i+j=d} A_i[k] B_j[k] <= 8 * 255^2 per k, so 16 k fit
// (8 * 255^2 * 16 = 8323200 < 2^23); then the 15 diagonals are combined into
// integers and the accumulators start again.
//
// One m16n8k16 MMA takes 8 k x 2 digits ("k8": thread t of a quad holds k = t and
// t + 4): A fragment i = digit pairs (2i, 2i + 1), B fragment e = digits (e, e - 1),
// which meet on diagonal 2i + e: 36 MMAs for 8 k.  For at most 4 k ("k4") the 16
// columns are 4 k x 4 digits: 22 MMAs.  Digits move by byte permutes only, one per
// fragment register (two for the pair that straddles the halves).
//
// Measured on GB300: mma.sync f16 runs at 996 multiply-adds per clock and SM; 64
// (k8: 72) of them replace four 32x32->64 integer multiply-adds of about 5 cycles
// per warp and sub-partition each.
#pragma once
#include "common.cuh"

namespace pencil {

constexpr u32 kDigitBias = 0x33000000u;   // bit pattern of 2^-25

// The start of an accumulator set: four registers, opaque to the compiler so that
// they stay one register quad for the whole kernel (a constant would be copied into
// every accumulator: 60 moves per set).
struct DigitZero {
  float z[4];
  __device__ __forceinline__ DigitZero() {
#pragma unroll
    for (int i = 0; i < 4; ++i) asm volatile("mov.b32 %0, 0x33000000;" : "=f"(z[i]));
  }
};

__device__ __forceinline__ void digit_mma(float (&d)[4], u32 a0, u32 a1, u32 a2, u32 a3, u32 b0, u32 b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void digit_mma_first(float (&d)[4], u32 a0, u32 a1, u32 a2, u32 a3, u32 b0, u32 b1,
                                                const DigitZero& z) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%12,%13};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(z.z[0]), "f"(z.z[1]), "f"(z.z[2]), "f"(z.z[3]));
}

// Digit pairs (2i, 2i + 1), i = 0 .. 3, of a word as two f16 subnormals each.
__device__ __forceinline__ void digit_pairs(u64 x, u32 (&p)[4]) {
  const u32 lo = (u32)x, hi = (u32)(x >> 32);
  p[0] = __byte_perm(lo, 0, 0x4140);
  p[1] = __byte_perm(lo, 0, 0x4342);
  p[2] = __byte_perm(hi, 0, 0x4140);
  p[3] = __byte_perm(hi, 0, 0x4342);
}

// Digits (e, e - 1), e = 0 .. 8 (digits -1 and 8 are zero).
__device__ __forceinline__ void digit_shifts(u64 x, u32 (&p)[9]) {
  const u32 lo = (u32)x, hi = (u32)(x >> 32);
  p[0] = lo & 0xFFu;
  p[1] = __byte_perm(lo, 0, 0x4041);
  p[2] = __byte_perm(lo, 0, 0x4142);
  p[3] = __byte_perm(lo, 0, 0x4243);
  p[4] = __byte_perm(lo, hi, 0x3344) & 0x00FF00FFu;
  p[5] = __byte_perm(hi, 0, 0x4041);
  p[6] = __byte_perm(hi, 0, 0x4142);
  p[7] = __byte_perm(hi, 0, 0x4243);
  p[8] = __byte_perm(hi, 0, 0x4344);
}

// acc[d] += diagonals of 8 k: words r0 / r1 = row g / g + 8 of k = t, r2 / r3 the
// same rows of k = t + 4; c0 / c1 = column g of k = t and t + 4 (g = lane / 4, t = lane % 4).
template <bool FIRST>
__device__ __forceinline__ void digits_k8(float (&acc)[15][4], u64 r0, u64 r1, u64 r2, u64 r3, u64 c0, u64 c1,
                                          const DigitZero& z) {
  u32 a0[4], a1[4], a2[4], a3[4], b0[9], b1[9];
  digit_pairs(r0, a0);
  digit_pairs(r1, a1);
  digit_pairs(r2, a2);
  digit_pairs(r3, a3);
  digit_shifts(c0, b0);
  digit_shifts(c1, b1);
#pragma unroll
  for (int e = 0; e < 9; ++e)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (FIRST && (e < 2 || i == 3))   // first product on diagonal 2i + e
        digit_mma_first(acc[2 * i + e], a0[i], a1[i], a2[i], a3[i], b0[e], b1[e], z);
      else
        digit_mma(acc[2 * i + e], a0[i], a1[i], a2[i], a3[i], b0[e], b1[e]);
    }
}

// The same for 4 k: words r0 / r1 = row g / g + 8 and c0 = column g of k = t.
template <bool FIRST>
__device__ __forceinline__ void digits_k4(float (&acc)[15][4], u64 r0, u64 r1, u64 c0,
                                          const DigitZero& z) {
  u32 a0[4], a1[4], b[9];
  digit_pairs(r0, a0);
  digit_pairs(r1, a1);
  digit_shifts(c0, b);
#pragma unroll
  for (int e = 0; e < 11; ++e)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const u32 x = e < 9 ? b[e] : 0u, y = e >= 2 ? b[e - 2] : 0u;
      if (FIRST && (e < 4 || i == 1))   // first product on diagonal 4i + e
        digit_mma_first(acc[4 * i + e], a0[2 * i], a1[2 * i], a0[2 * i + 1], a1[2 * i + 1], x, y, z);
      else
        digit_mma(acc[4 * i + e], a0[2 * i], a1[2 * i], a0[2 * i + 1], a1[2 * i + 1], x, y);
    }
}

// Constants of one prime q = 2^b - c for the folds below.
struct DigitMod {
  u32 c64, c, sb, m;   // 2^64 mod q, c, b - 32, 2^(b-32) - 1
  __device__ __forceinline__ explicit DigitMod(const LimbConst& lc)
      : c64((u32)lc.c64), c((u32)lc.cb), sb(lc.sb), m((1u << lc.sb) - 1u) {}
};

// The 15 diagonals of output o of an accumulator set, combined modulo q.  With
// b_d the bit patterns, P_j = b_2j + 2^8 b_(2j+1) mod 2^32 drops the odd diagonals'
// bias (kDigitBias 2^8 = 0 mod 2^32) and does not wrap; S' = sum_j P_j 2^(16 j),
// j = 0 .. 6, plus the last diagonal without its bias, = S + kDigitBias sum_j 2^(16 j)
// < 2^127 (operands below 2^61).  Even P_j are words of S', odd ones straddle two:
// four byte permutes and one 128-bit addition.  Then 2^64 = c64 (< 2^32) and
// 2^b = c (< 2^(b-32)) mod q fold S' to a value below 2^63 + 2^61 congruent to
// S + bias; the caller folds it once more (fold_b) before it sums several, and
// subtracts the bias of all its combinations at once.
// One PTX block: as C the 64-bit addends assembled from 32-bit halves cost moves.
__device__ __forceinline__ u64 digits_mod(const float (&acc)[15][4], int o, const DigitMod& q) {
  u64 r;
  asm("{\n\t"
      ".reg .u32 p0, p1, p2, p3, p4, p5, p6, x, y, z, w, a0, a1, a2, a3, l, h, s;\n\t"
      ".reg .u64 t, v;\n\t"
      "mad.lo.u32 p0, %2, 256, %1;\n\t"
      "mad.lo.u32 p1, %4, 256, %3;\n\t"
      "mad.lo.u32 p2, %6, 256, %5;\n\t"
      "mad.lo.u32 p3, %8, 256, %7;\n\t"
      "mad.lo.u32 p4, %10, 256, %9;\n\t"
      "mad.lo.u32 p5, %12, 256, %11;\n\t"
      "mad.lo.u32 p6, %14, 256, %13;\n\t"
      "mad.lo.u32 p6, %15, 65536, p6;\n\t"
      "shl.b32 x, p1, 16;\n\t"
      "prmt.b32 y, p1, p3, 0x5432;\n\t"
      "prmt.b32 z, p3, p5, 0x5432;\n\t"
      "shr.u32 w, p5, 16;\n\t"
      "add.cc.u32 a0, p0, x;\n\t"
      "addc.cc.u32 a1, p2, y;\n\t"
      "addc.cc.u32 a2, p4, z;\n\t"
      "addc.u32 a3, p6, w;\n\t"
      "mul.wide.u32 t, a2, %16;\n\t"
      "mov.b64 {l, h}, t;\n\t"
      "mul.wide.u32 t, a3, %16;\n\t"
      "add.cc.u32 a0, a0, l;\n\t"
      "addc.cc.u32 a1, a1, h;\n\t"
      "mov.b64 {l, h}, t;\n\t"
      "addc.u32 h, h, 0;\n\t"
      "add.cc.u32 a1, a1, l;\n\t"
      "addc.u32 h, h, 0;\n\t"
      "shr.u32 s, a1, %18;\n\t"
      "and.b32 a1, a1, %19;\n\t"
      "mov.b64 v, {a0, a1};\n\t"
      "mad.wide.u32 v, h, %16, v;\n\t"
      "mad.wide.u32 %0, s, %17, v;\n\t"
      "}"
      : "=l"(r)
      : "r"(__float_as_uint(acc[0][o])), "r"(__float_as_uint(acc[1][o])), "r"(__float_as_uint(acc[2][o])),
        "r"(__float_as_uint(acc[3][o])), "r"(__float_as_uint(acc[4][o])), "r"(__float_as_uint(acc[5][o])),
        "r"(__float_as_uint(acc[6][o])), "r"(__float_as_uint(acc[7][o])), "r"(__float_as_uint(acc[8][o])),
        "r"(__float_as_uint(acc[9][o])), "r"(__float_as_uint(acc[10][o])), "r"(__float_as_uint(acc[11][o])),
        "r"(__float_as_uint(acc[12][o])), "r"(__float_as_uint(acc[13][o])), "r"(__float_as_uint(acc[14][o])),
        "r"(q.c64), "r"(q.c), "r"(q.sb), "r"(q.m));
  return r;
}

// v mod q, lazily: any v < 2^64 -> below 2^b + 2^32.
__device__ __forceinline__ u64 fold_b(u64 v, const DigitMod& q) {
  u64 r;
  asm("{\n\t"
      ".reg .u32 l, h, s;\n\t.reg .u64 t;\n\t"
      "mov.b64 {l, h}, %1;\n\t"
      "shr.u32 s, h, %3;\n\t"
      "and.b32 h, h, %4;\n\t"
      "mov.b64 t, {l, h};\n\t"
      "mad.wide.u32 %0, s, %2, t;\n\t"
      "}"
      : "=l"(r)
      : "l"(v), "r"(q.c), "r"(q.sb), "r"(q.m));
  return r;
}

}  // namespace pencil
