// The NTT-domain ct x pt multiply-accumulate (Alg. 1 step 2 / Alg. 2 step 2) as a
// batch of small matrix products on the tensor cores: for every slot (limb,
// coefficient), out[m, c][n] = sum_k A_c[m, k] B[k, n] (+ A'[m, k] B'_c[k, n]) mod q_j,
// exactly (digits.cuh).
//
// CTA = 4 consecutive slots (32 bytes of every operand row) of an output block of
// MT rows m x NT columns n; warp w = slot w.  The 16 rows of an MMA tile are output
// columns n, its 8 columns are 4 rows m x 2 components (Alg. 2: 8 rows m of one
// component, because the second product's ciphertext is B').  Input blocks k come
// in chunks of 16 (Alg. 2: 8) through one or two shared-memory stages (16-byte
// cp.async; the next chunk is copied while the current one is multiplied).  The sums
// of one chunk fit the f32 accumulators, so a tile's registers hold no state between
// chunks: its 128 outputs are combined modulo q once per chunk and summed lazily in
// shared memory, from where they are re-masked and stored in row segments.
//
// What bounds it (ncu, conv3x3 128->128, M = 32, K = 43, NC = 64, L N = 24576, 88064
// products: 2.25 ms, integer kernel 4.02 ms): tensor pipe 48 % busy, issue 51 %; a
// tile's combination (142 of its ~400 instructions) waits for its last MMA, and 16
// warps per SM (109 registers, 60 of them accumulators) overlap the two only partly.
// M = 10, K = 16, NC = 16 (2560 products): 96 us against 139 us.  Variants measured
// and not kept: 8 slots per CTA of 8 warps (108 us: coarser barriers), persistent
// CTAs with the next block's copies in flight (131 us), 16 x 32 blocks with K > 16
// (1 CTA per SM).
#pragma once
#include "digits.cuh"
#include "kernels.h"

namespace pencil {

#define MMA_LANES 4
#define MMA_THREADS (32 * MMA_LANES)
#define MMA_R8 (8 * MMA_LANES)   // words of 8 rows

__device__ __forceinline__ void mma_cp16(u64* smem, const u64* gmem, int bytes) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(bytes) : "memory");
}

// Shared memory of an output block of MT rows m (Alg. 2: at least 8) x NT columns n.
// Rows (one k of one operand row) are 4 slots = 32 bytes; the slot pairs of a row are
// swapped by the row number's bit 2, so the rows of a fragment (8 consecutive row
// numbers) hit 8 distinct 16-byte bank groups.  Stage regions:
// B (Alg. 2: B, B'_0, B'_1), A (both components), NTT(Delta x0) or A'.
template <bool DUAL, int MT, int NT>
struct MmaTile {
  static constexpr int KC = DUAL ? 8 : 16;   // input blocks of a chunk
  static constexpr int RB = KC * NT, RA = KC * 2 * MT, RP = KC * MT;   // rows of a region
  static constexpr int NB = DUAL ? 3 : 1;
  static constexpr int STAGE = (NB * RB + RA + RP) * MMA_LANES;                    // words
  // one slot's output sums: 128 per unit (tile of 16 n x 8 columns); 4 mod 8 words apart
  static constexpr int SUMS = (NT / 16) * (MT / 4) * 128 + 4;
  static constexpr size_t bytes(int stages) { return (size_t)(stages * STAGE + MMA_LANES * SUMS) * sizeof(u64); }
};

__device__ __forceinline__ int mma_word(int row, int chunk) {   // word of slot pair `chunk` of a row
  return row * MMA_LANES + ((chunk ^ ((row >> 2) & 1)) << 1);
}

// Copies rows (k, i), k < kpad, i < ni of an n- or m-indexed region of I rows per k:
// row (k, i) = src + k kstep + i istep (4 slots).  Rows i >= ni are left alone (their
// outputs are not stored); rows k >= kc are zeroed when ZERO, else left alone (the
// other operand's are zero).
template <int I, int KC, bool ZERO>
__device__ __forceinline__ void mma_copy(u64* dst, const u64* src, size_t kstep, size_t istep, int ni, int kc,
                                         int kpad) {
  const int chunk = threadIdx.x & 1, r0 = threadIdx.x >> 1;   // 64 rows per pass of the CTA
  const int i = r0 & (I - 1), k0 = r0 / I;
  constexpr int DK = 64 / I;
  if (i >= ni) return;
  const u64* g = src + (size_t)k0 * kstep + (size_t)i * istep + 2 * chunk;
#pragma unroll
  for (int p = 0; p < (KC + DK - 1) / DK; ++p, g += DK * kstep) {
    const int k = k0 + p * DK;
    const int row = ((k >> 2) * (I / 2) + (i >> 1)) * 8 + (i & 1) * 4 + (k & 3);
    if (k < kc)
      mma_cp16(dst + mma_word(row, chunk), g, 16);
    else if (ZERO && k < kpad)
      mma_cp16(dst + mma_word(row, chunk), src, 0);
  }
}

template <bool DUAL, int MT, int NT>
__device__ __forceinline__ void mma_issue(const MacParams& P, int m0, int n0, int k0, int lane0, u64* st) {
  using T = MmaTile<DUAL, MT, NT>;
  const int kc = min(T::KC, P.K - k0), kpad = (kc + 3) & ~3;
  const int nn = min(NT, P.NC - n0), mm = min(MT, P.M - m0);
  const size_t kn = (size_t)k0 * P.NC + n0, mk = (size_t)m0 * P.K + k0;
  u64* a = st + T::NB * T::RB * MMA_LANES;
  u64* p = a + T::RA * MMA_LANES;
  mma_copy<NT, T::KC, true>(st, P.b + kn * P.b_stride + lane0, (size_t)P.NC * P.b_stride, P.b_stride, nn, kc, kpad);
  if constexpr (DUAL) {
    // columns: component c in its own half
    const size_t ak = (size_t)P.K * P.a0_stride;
    mma_copy<MT, T::KC, false>(a, P.a0 + mk * P.a0_stride + lane0, P.a0_stride, ak, mm, kc, kpad);
    mma_copy<MT, T::KC, false>(a + T::RP * MMA_LANES, P.a1 + mk * P.a0_stride + lane0, P.a0_stride, ak, mm, kc, kpad);
    mma_copy<MT, T::KC, false>(p, P.pa + mk * P.pa_stride + lane0, P.pa_stride, (size_t)P.K * P.pa_stride, mm, kc, kpad);
    const size_t ck = (size_t)P.NC * P.cb_stride;
    mma_copy<NT, T::KC, true>(st + T::RB * MMA_LANES, P.cb0 + kn * P.cb_stride + lane0, ck, P.cb_stride, nn, kc, kpad);
    mma_copy<NT, T::KC, true>(st + 2 * T::RB * MMA_LANES, P.cb1 + kn * P.cb_stride + lane0, ck, P.cb_stride, nn, kc, kpad);
  } else {
    const int chunk = threadIdx.x & 1, r0 = threadIdx.x >> 1;
    {   // column 2 i + c = component c of row m0 + i
      const int col = r0 & (2 * MT - 1), i = col >> 1, kb = r0 / (2 * MT);
      constexpr int DK = 64 / (2 * MT);
      if (i < mm) {
        const u64* g = ((col & 1) ? P.a1 : P.a0) + (mk + (size_t)i * P.K + kb) * P.a0_stride + lane0 + 2 * chunk;
#pragma unroll
        for (int q = 0; q < (T::KC + DK - 1) / DK; ++q, g += DK * P.a0_stride) {
          const int k = kb + q * DK, row = ((k >> 2) * MT + i) * 8 + (col & 1) * 4 + (k & 3);
          if (k < kc) mma_cp16(a + mma_word(row, chunk), g, 16);
        }
      }
    }
    if (P.p0) {   // NTT(Delta x0)[m, k]: rows ((k / 4) MT + i) 4 + k % 4
      const int i = r0 & (MT - 1), kb = r0 / MT;
      constexpr int DK = 64 / MT;
      if (i < mm) {
        const u64* g = P.p0 + (mk + (size_t)i * P.K + kb) * P.p0_stride + lane0 + 2 * chunk;
#pragma unroll
        for (int q = 0; q < (T::KC + DK - 1) / DK; ++q, g += DK * P.p0_stride) {
          const int k = kb + q * DK, row = ((k >> 2) * MT + i) * 4 + (k & 3);
          if (k < kc) mma_cp16(p + mma_word(row, chunk), g, 16);
        }
      }
    }
  }
  if (k0 == 0 && P.mask) {   // the re-mask rows the block's store reads: into L2 now, not from DRAM at the end
    const int n = threadIdx.x & (NT - 1);
    for (int m = threadIdx.x / NT; m < mm; m += MMA_THREADS / NT)
      if (n < nn)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(P.mask + ((size_t)(m0 + m) * P.NC + n0 + n) * (size_t)P.lanes +
                                                      lane0));
  }
}

// One chunk (input blocks [k0, k0 + KC)) of an output block: warp w = slot w.
template <bool DUAL, int MT, int NT>
__device__ __forceinline__ void mma_chunk(const u64* st, u64* sums, const DigitMod& qd, const DigitZero& zero, int kc,
                                          int ch, bool single, int its, int cts, bool has_p) {
  using T = MmaTile<DUAL, MT, NT>;
  const int w = threadIdx.x >> 5, ln = threadIdx.x & 31, g = ln >> 2, t = ln & 3;
  // this thread's word of a fragment row: rows 8 x + 4 (g & 1) + t of slot w
  const int fo = mma_word((g & 1) * 4 + t, w >> 1) + (w & 1);
  const int po = mma_word(((g >> 1) & 1) * 4 + t, w >> 1) + (w & 1);
  const bool addp = has_p && !(g & 1);
  u64* sum = sums + w * T::SUMS + ln;
  const u64* fb = st + (g >> 1) * MMA_R8 + fo;
  const u64* fa0 = st + T::NB * T::RB * MMA_LANES + (g >> 1) * MMA_R8 + fo;
  const u64* fp0 = st + (T::NB * T::RB + T::RA) * MMA_LANES + (DUAL ? (g >> 1) * MMA_R8 + fo : (g >> 2) * MMA_R8 + po);
  const bool first = ch == 0, fold = (ch & 7) == 7;
  float acc[15][4];
  for (int it = 0; it < its; ++it, fb += 8 * MMA_R8) {
    constexpr int BN = NT / 2 * MMA_R8, B8 = 4 * MMA_R8;   // four k further
#pragma unroll 1
    for (int c = 0; c < (DUAL ? 2 : 1); ++c) {
      const u64* fa = fa0 + c * T::RP * MMA_LANES;
      const u64* fp = fp0;
#pragma unroll 1
      for (int ct = 0; ct < cts; ++ct, sum += 128, fa += 4 * MMA_R8, fp += (DUAL ? 4 : 2) * MMA_R8) {
        if constexpr (DUAL) {
          constexpr int BA = MT / 2 * MMA_R8;
          const u64* fc = fb + (1 + c) * T::RB * MMA_LANES;
          if (kc > 4) {
            digits_k8<true>(acc, fb[0], fb[B8], fb[BN], fb[BN + B8], fa[0], fa[BA], zero);
            digits_k8<false>(acc, fc[0], fc[B8], fc[BN], fc[BN + B8], fp[0], fp[BA], zero);
          } else {
            digits_k4<true>(acc, fb[0], fb[B8], fa[0], zero);
            digits_k4<false>(acc, fc[0], fc[B8], fp[0], zero);
          }
        } else {
          constexpr int BA = MT * MMA_R8, BP = MT / 2 * MMA_R8;
          auto col = [&](int j) {   // column g of k = 4 j + t: c0 + NTT(Delta x0), or c1
            u64 v = fa[j * BA];
            if (addp) v += fp[j * BP];
            return v;
          };
          if (kc > 4)
            digits_k8<true>(acc, fb[0], fb[B8], fb[BN], fb[BN + B8], col(0), col(1), zero);
          else
            digits_k4<true>(acc, fb[0], fb[B8], col(0), zero);
          if (kc > 12)
            digits_k8<false>(acc, fb[2 * BN], fb[2 * BN + B8], fb[3 * BN], fb[3 * BN + B8], col(2), col(3), zero);
          else if (kc > 8)
            digits_k4<false>(acc, fb[2 * BN], fb[2 * BN + B8], col(2), zero);
        }
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          u64 v = digits_mod(acc, o, qd);
          if (!single) {
            v = fold_b(v, qd);
            if (!first) v += sum[o * 32];
            if (fold) v = fold_b(v, qd);
          }
          sum[o * 32] = v;
        }
      }
    }
  }
}

// Sums of a finished block -> canonical, re-mask, 32-byte row segments: thread = slot
// pair 2 chunk of outputs (fragment lane l2, output o), o = o1 and o1 + 2 (columns n
// and n + 8) of every unit.
template <bool DUAL, int MT, int NT>
__device__ __forceinline__ void mma_store(const MacParams& P, const u64* sums, const DigitMod& qd, u64 q, u64 start,
                                          int m0, int n0, int lane0, int its, int cts) {
  using T = MmaTile<DUAL, MT, NT>;
  const int tid = threadIdx.x, chunk = tid & 1, l2 = (tid >> 1) & 31, o1 = tid >> 6;
  const size_t lnw = (size_t)P.lanes;
  const int mm = min(MT, P.M - m0);
  const u64* s0 = sums + (2 * chunk) * T::SUMS + o1 * 32 + l2;
  const int mcol = DUAL ? (l2 & 3) * 2 + o1 : (l2 & 3);   // row m within the column tile
  const int n = n0 + (l2 >> 2);
  const size_t mn = (size_t)(m0 + mcol) * P.NC + n, col = (size_t)P.NC * lnw;   // words between output rows
  const u64* km = P.mask + mn * lnw + lane0 + 2 * chunk;
  u64* dst = P.out + (2 * mn + (DUAL ? 0 : o1)) * lnw + lane0 + 2 * chunk;
  const bool masked = P.mask != nullptr;
  constexpr int MC = DUAL ? 8 : 4;   // rows m of a column tile
  for (int it = 0; it < its; ++it, km += 16 * lnw, dst += 32 * lnw) {
    const int left = P.NC - n - 16 * it;   // columns n, n + 8 exist when left > 0, > 8
#pragma unroll 1
    for (int c = 0; c < (DUAL ? 2 : 1); ++c) {
      const u64* kp = km;
      u64* dp = dst + c * lnw;
      const bool sub = masked && (DUAL ? c == 0 : o1 == 0);
#pragma unroll 1
      for (int ct = 0; ct < cts; ++ct, s0 += 128, kp += MC * col, dp += 2 * MC * col) {
        if (ct * MC + mcol >= mm) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (left <= 8 * j) continue;
          u64 v0 = s0[j * 64] + start, v1 = s0[T::SUMS + j * 64] + start;
          if (sub) {
            const ulonglong2 k = __ldg(reinterpret_cast<const ulonglong2*>(kp + j * 8 * lnw));
            v0 += q - k.x;
            v1 += q - k.y;
          }
          v0 = csub(fold_b(v0, qd), q);
          v1 = csub(fold_b(v1, qd), q);
          *reinterpret_cast<ulonglong2*>(dp + j * 16 * lnw) = make_ulonglong2(v0, v1);
        }
      }
    }
  }
}

// One output block (rows [m0, m0 + MT), columns [n0, n0 + NT)) of slots lane0 .. + 3.
// MMA_THREADS threads; smem of MmaTile::bytes(2), or bytes(1) when K <= KC.
template <bool DUAL, int MT, int NT>
__device__ __forceinline__ void mac_mma_block(const DevCtx& ctx, const MacParams& P, int m0, int n0, int lane0,
                                              u64* sm) {
  using T = MmaTile<DUAL, MT, NT>;
  const int chunks = (P.K + T::KC - 1) / T::KC;
  u64* sums = sm + (chunks > 1 ? 2 : 1) * T::STAGE;
  const DigitZero zero;
  const int limb = lane0 >> ctx.log_n;
  const DigitMod qd(ctx.limb[limb]);
  const int its = (min(NT, P.NC - n0) + 15) >> 4;
  const int mm = min(MT, P.M - m0), cts = DUAL ? (mm + 7) >> 3 : (mm + 3) >> 2;   // (Alg. 2: of each component)
  mma_issue<DUAL, MT, NT>(P, m0, n0, 0, lane0, sm);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  for (int ch = 0; ch < chunks; ++ch) {
    if (ch + 1 < chunks)
      mma_issue<DUAL, MT, NT>(P, m0, n0, (ch + 1) * T::KC, lane0, sm + ((ch + 1) & 1) * T::STAGE);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    mma_chunk<DUAL, MT, NT>(sm + (ch & 1) * T::STAGE, sums, qd, zero, min(T::KC, P.K - ch * T::KC), ch, chunks == 1,
                            its, cts, !DUAL && P.p0 != nullptr);
    __syncthreads();   // the stage may be refilled; after the last chunk: every sum is written
  }
  mma_store<DUAL, MT, NT>(P, sums, qd, ctx.limb[limb].q, P.start[limb], m0, n0, lane0, its, cts);
}

}  // namespace pencil
