// Plaintext correlations over Z_t (t = 2^t_bits) on the tensor cores:
//   out[a, o, i, j] = addends + sum_{c, u, v} W(o, c, u, v) V(a, c, i + u, j + v)  mod t
// as one matrix product, rows o, columns (a, i, j), reduction k = (c, u, v), in exact
// base-256 digits (digits.cuh).  Only the diagonals below 8 D >= t_bits matter: 12
// (D = 6) or 20 (D = 8) MMAs per 8 k of a 16 x 8 tile; after 16 k they are combined
// modulo 2^64 and added to a tile's 64-bit sums in registers.
//
// CTA = 4 warps on BM rows x BN columns; chunks of 16 k of both operands arrive as
// 64-bit words by 8-byte cp.async (zero-filled outside the input), three stages, two
// in flight.  A thread's words are spread along k or along rows, whichever is
// contiguous in memory for that operand.  A reduction long against the number of
// tiles is split over the grid: the output starts as the sum of the addends, every
// part adds its sums with 64-bit atomics (addition mod 2^64 is exact in any order)
// and a last pass masks.
//
// What bounds it: 64-bit low products on the integer pipe ran at 0.96 T multiply-adds
// per second (grad_W of conv3x3 128->128, 16x16, batch 128: 4.99 ms); here the same
// takes 0.78 ms, the tensor pipe 53 % busy (ncu): two 4-warp CTAs per SM (255
// registers, 64 of them sums) overlap extraction and combination with the MMAs only
// partly.  conv3x3 16->16, 32x32, batch 512: 534 -> 260 us (37 %: 18 loads per thread
// and chunk for 4 tiles); fc 2048->1001, batch 64: 1608 -> 42 us.
#include <algorithm>

#include "digits.cuh"
#include "kernels.h"
#include "rules.h"

namespace pencil {

#define RM_KC 16           // (ring_split's chunks)
#define RM_PITCH 18        // words of a row of 16 k: 144 bytes, LDS.128 of 8 rows x 4 threads conflict-free
#define RM_STAGES 3
#define RM_THREADS 128

struct RingMma {
  long long npos;          // B * Ho * Wo
  long long K;             // reduction length of this launch, from element k0 on
  long long k0;
  int chunks, per;         // chunks of 16, chunks of one part
  int v_rows, w_rows;      // lanes along rows (1) or along k (0)
  int split;               // several parts or launches: atomics
};

struct RmRow {   // one output column (position) of V: offset of its window, window origin
  i64 off;
  int i, j;
};
struct RmK {     // one k: offset into V and the kernel position (u far outside when k >= K)
  i64 v;
  int u, x;
};

__device__ __forceinline__ void rm_cp8(u64* smem, const u64* gmem, bool ok) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(ok ? 8 : 0) : "memory");
}

template <int D>
__device__ __forceinline__ void rm_pairs(u64 x, u32 (&p)[D / 2]) {
  const u32 lo = (u32)x, hi = (u32)(x >> 32);
  p[0] = __byte_perm(lo, 0, 0x4140);
  p[1] = __byte_perm(lo, 0, 0x4342);
  p[2] = __byte_perm(hi, 0, 0x4140);
  if constexpr (D > 6) p[3] = __byte_perm(hi, 0, 0x4342);
}
template <int D>
__device__ __forceinline__ void rm_shifts(u64 x, u32 (&p)[D]) {
  const u32 lo = (u32)x, hi = (u32)(x >> 32);
  p[0] = lo & 0xFFu;
  p[1] = __byte_perm(lo, 0, 0x4041);
  p[2] = __byte_perm(lo, 0, 0x4142);
  p[3] = __byte_perm(lo, 0, 0x4243);
  p[4] = __byte_perm(lo, hi, 0x3344) & 0x00FF00FFu;
  p[5] = __byte_perm(hi, 0, 0x4041);
  if constexpr (D > 6) {
    p[6] = __byte_perm(hi, 0, 0x4142);
    p[7] = __byte_perm(hi, 0, 0x4243);
  }
}

// sum += the D diagonals of output o, with kDigitBias (1 + 2^16 + .. ) extra (digits_mod
// explains the even / odd diagonals' bias).
template <int D>
__device__ __forceinline__ void rm_add(u64& sum, const float (&acc)[D][4], int o) {
  u32 p[D / 2];
#pragma unroll
  for (int j = 0; j < D / 2; ++j) p[j] = __float_as_uint(acc[2 * j][o]) + (__float_as_uint(acc[2 * j + 1][o]) << 8);
  u32 hi = (p[1] >> 16) + p[2];
  if constexpr (D > 6) hi += p[3] << 16;
  sum += (((u64)hi) << 32) | (p[1] << 16);
  sum += p[0];
}

template <int D, int MI, int WM, int WN>
__global__ void __launch_bounds__(RM_THREADS, MI == 2 ? 2 : 3) k_ring_mma(const __grid_constant__ RingParams P,
                                                            const __grid_constant__ RingMma R) {
  constexpr int BM = 16 * MI * WM, BN = 32 * WN;
  static_assert(WM * WN == 4, "four warps");
  extern __shared__ __align__(16) u64 sm[];   // [RM_STAGES][BM + BN][RM_PITCH]
  __shared__ __align__(16) RmRow rows[BN];
  __shared__ __align__(16) RmK ktab[2][RM_KC];
  __shared__ i64 kw[2][RM_KC];                // offset of k into W
  const int tid = threadIdx.x, warp = tid >> 5, ln = tid & 31, g = ln >> 2, t = ln & 3;
  const int wm = warp / WN, wn = warp % WN;
  const long long pos0 = (long long)blockIdx.x * BN;
  const int o0 = blockIdx.y * BM;
  const int Co = P.kbound.x, KH = P.kbound.z, KW = P.kbound.w;
  const int c0 = blockIdx.z * R.per, c1 = min(R.chunks, c0 + R.per);
  constexpr int FAR = -(1 << 30);
  if (tid < BN) {
    const long long pos = pos0 + tid;
    RmRow r{0, FAR, FAR};
    if (pos < R.npos) {
      const int hw = P.Ho * P.Wo;
      const long long a = pos / hw;
      const int rem = (int)(pos - a * hw), i = rem / P.Wo, j = rem - i * P.Wo;
      r.i = i - P.v.pr;
      r.j = j - P.v.ps;
      r.off = P.v.base + a * P.v.s0 + (i64)r.i * P.v.s2 + (i64)r.j * P.v.s3;
    }
    rows[tid] = r;
  }
  auto make_k = [&](int ch) {   // threads 0 .. 15
    const long long k = (long long)ch * RM_KC + tid;
    RmK e{0, FAR, 0};
    i64 w = 0;
    if (k < R.K) {
      const long long uv = (long long)KH * KW, e0 = R.k0 + k, c = e0 / uv;
      const int q = (int)(e0 - c * uv);
      e.u = q / KW;
      e.x = q - e.u * KW;
      e.v = c * P.v.s1 + e.u * P.v.s2 + e.x * P.v.s3;
      w = P.w.base + c * P.w.s1 + e.u * P.w.s2 + e.x * P.w.s3;
    }
    ktab[ch & 1][tid] = e;
    kw[ch & 1][tid] = w;
  };
  auto issue = [&](int ch) {
    u64* st = sm + (ch % RM_STAGES) * ((BM + BN) * RM_PITCH);
    const RmK* kt = ktab[ch & 1];
    // in row order a thread's row, in k order its k, is the same in every pass
    if (R.w_rows) {   // W: rows o
      const int r = tid % BM;
      const u64* src = P.w.ptr + (i64)(o0 + r) * P.w.s0;
      const bool in = o0 + r < Co;
      u64* dst = st + r * RM_PITCH;
#pragma unroll
      for (int p = 0; p < BM / 8; ++p) {
        const int kk = tid / BM + p * (RM_THREADS / BM);
        const bool ok = in && (long long)ch * RM_KC + kk < R.K;
        rm_cp8(dst + kk, ok ? src + kw[ch & 1][kk] : P.w.ptr, ok);
      }
    } else {
      const int kk = tid & 15, r0 = tid >> 4;
      const bool in = (long long)ch * RM_KC + kk < R.K;
      const u64* src = P.w.ptr + kw[ch & 1][kk] + (i64)(o0 + r0) * P.w.s0;
      u64* dst = st + r0 * RM_PITCH + kk;
#pragma unroll
      for (int p = 0; p < BM / 8; ++p, src += 8 * P.w.s0) {
        const bool ok = in && o0 + r0 + 8 * p < Co;
        rm_cp8(dst + 8 * p * RM_PITCH, ok ? src : P.w.ptr, ok);
      }
    }
    u64* sv = st + BM * RM_PITCH;
    if (R.v_rows) {   // V: columns (a, i, j)
      const int r = tid % BN;
      const RmRow row = rows[r];
      const u64* src = P.v.ptr + row.off;
      u64* dst = sv + r * RM_PITCH;
#pragma unroll
      for (int p = 0; p < BN / 8; ++p) {
        const int kk = tid / BN + p * (RM_THREADS / BN);
        const RmK k = kt[kk];
        const bool ok = (unsigned)(row.i + k.u) < (unsigned)P.v.hr && (unsigned)(row.j + k.x) < (unsigned)P.v.wr;
        rm_cp8(dst + kk, ok ? src + k.v : P.v.ptr, ok);
      }
    } else {
      const int kk = tid & 15, r0 = tid >> 4;
      const RmK k = kt[kk];
      const u64* src = P.v.ptr + k.v;
      u64* dst = sv + r0 * RM_PITCH + kk;
#pragma unroll
      for (int p = 0; p < BN / 8; ++p) {
        const RmRow row = rows[r0 + 8 * p];
        const bool ok = (unsigned)(row.i + k.u) < (unsigned)P.v.hr && (unsigned)(row.j + k.x) < (unsigned)P.v.wr;
        rm_cp8(dst + 8 * p * RM_PITCH, ok ? src + row.off : P.v.ptr, ok);
      }
    }
  };
  if (tid < RM_KC) {
    make_k(c0);
    make_k(c0 + 1);
  }
  __syncthreads();
  issue(c0);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  if (c0 + 1 < c1) issue(c0 + 1);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  __syncthreads();   // the table slot of chunk c0 is free
  if (tid < RM_KC) make_k(c0 + 2);

  const DigitZero zero;
  u64 sum[MI][4][4];
#pragma unroll
  for (int mi = 0; mi < MI; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni)
#pragma unroll
      for (int o = 0; o < 4; ++o) sum[mi][ni][o] = 0;

  for (int ch = c0; ch < c1; ++ch) {
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();   // chunk ch is here; chunk ch - 1 has been read; the table of ch + 2 is written
    if (ch + 2 < c1) issue(ch + 2);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (tid < RM_KC) make_k(ch + 3);
    const u64* st = sm + (ch % RM_STAGES) * ((BM + BN) * RM_PITCH);
    const u64* sv = st + (BM + wn * 32 + g) * RM_PITCH + 4 * t;
#pragma unroll
    for (int mi = 0; mi < MI; ++mi) {
      // thread t of a quad owns k = 4 t .. 4 t + 3 of the chunk (the same in both operands)
      u32 a[4][2][D / 2];   // [k][row g, g + 8][digit pair]
      {
        const u64* ra = st + ((wm * MI + mi) * 16 + g) * RM_PITCH + 4 * t;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(ra + h * 8 * RM_PITCH);
          const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(ra + h * 8 * RM_PITCH + 2);
          rm_pairs<D>(x.x, a[0][h]);
          rm_pairs<D>(x.y, a[1][h]);
          rm_pairs<D>(y.x, a[2][h]);
          rm_pairs<D>(y.y, a[3][h]);
        }
      }
#pragma unroll
      for (int ni = 0; ni < 4; ++ni) {
        const u64* rb = sv + ni * 8 * RM_PITCH;
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(rb);
        const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(rb + 2);
        float acc[D][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          u32 b0[D], b1[D];
          rm_shifts<D>(h ? y.x : x.x, b0);
          rm_shifts<D>(h ? y.y : x.y, b1);
#pragma unroll
          for (int e = 0; e < D; ++e)
#pragma unroll
            for (int i = 0; i < D / 2; ++i) {
              if (2 * i + e >= D) continue;
              if (h == 0 && e < 2)
                digit_mma_first(acc[2 * i + e], a[2 * h][0][i], a[2 * h][1][i], a[2 * h + 1][0][i], a[2 * h + 1][1][i],
                                b0[e], b1[e], zero);
              else
                digit_mma(acc[2 * i + e], a[2 * h][0][i], a[2 * h][1][i], a[2 * h + 1][0][i], a[2 * h + 1][1][i],
                          b0[e], b1[e]);
            }
        }
#pragma unroll
        for (int o = 0; o < 4; ++o) rm_add<D>(sum[mi][ni][o], acc, o);
      }
    }
  }
  // minus the bias of all combinations; outputs (o, position) at their flat indices
  const u64 one = (u64)kDigitBias * (1ull + (1ull << 16) + (1ull << 32) + (D > 6 ? 1ull << 48 : 0ull));
  const u64 bias = one * (u64)(c1 - c0);
#pragma unroll
  for (int ni = 0; ni < 4; ++ni)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int r = wn * 32 + ni * 8 + 2 * t + w;
      const long long pos = pos0 + r;
      if (pos >= R.npos) continue;
      const int hw = P.Ho * P.Wo;
      const long long a = pos / hw;
      const int i = rows[r].i + P.v.pr, j = rows[r].j + P.v.ps;
      const i64 base = P.y.base + a * P.y.s0 + i * P.y.s2 + j * P.y.s3;
#pragma unroll
      for (int mi = 0; mi < MI; ++mi)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int o = o0 + (wm * MI + mi) * 16 + g + 8 * h;
          if (o >= Co) continue;
          const i64 flat = base + o * P.y.s1;
          u64 v = sum[mi][ni][2 * h + w] - bias;
          if (R.split) {
            atomicAdd(reinterpret_cast<unsigned long long*>(P.out + flat), (unsigned long long)v);
          } else {
            if (P.addend) v += P.addend[flat];
            if (P.addend2) v += P.addend2[flat];
            P.out[flat] = v & P.t_mask;
          }
        }
    }
}

// First and last pass of a split reduction: out = addends (init), out &= t_mask.
__global__ void __launch_bounds__(256) k_ring_edge(RingParams P, int init) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= P.outs) return;
  if (!init) {
    P.out[e] &= P.t_mask;
    return;
  }
  u64 v = 0;
  if (P.addend) v += P.addend[e];
  if (P.addend2) v += P.addend2[e];
  P.out[e] = v;
}

template <int D, int MI, int WM, int WN>
static cudaError_t launch(const RingParams& P, RingMma R, int sms, cudaStream_t s) {
  constexpr int BM = 16 * MI * WM, BN = 32 * WN;
  constexpr size_t smem = (size_t)RM_STAGES * (BM + BN) * RM_PITCH * sizeof(u64);
  cudaError_t e =
      cudaFuncSetAttribute(k_ring_mma<D, MI, WM, WN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long gx = (R.npos + BN - 1) / BN, gy = (P.kbound.x + BM - 1) / BM;
  const long long K = R.K;
  R.split = K > kRingLaunchK || ring_split(K, gx * gy, sms).parts > 1;
  const unsigned eb = (unsigned)((P.outs + 255) / 256);
  if (R.split) {
    k_ring_edge<<<eb, 256, 0, s>>>(P, 1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  for (R.k0 = 0; R.k0 < K; R.k0 += kRingLaunchK) {
    R.K = std::min(K - R.k0, kRingLaunchK);
    const RingSplit r = ring_split(R.K, gx * gy, sms);
    R.chunks = r.chunks;
    R.per = r.per;
    k_ring_mma<D, MI, WM, WN><<<dim3((unsigned)gx, (unsigned)gy, (unsigned)r.parts), RM_THREADS, smem, s>>>(P, R);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (R.split) {
    k_ring_edge<<<eb, 256, 0, s>>>(P, 0);
    e = cudaGetLastError();
  }
  return e;
}

// Words of a warp's load that are contiguous: along output columns (rows of V), output
// channels (rows of W), or the reduction.
static int run(long long inner, i64 s_inner, long long outer, i64 s_outer) {
  if (inner > 1) return s_inner == 1 || s_inner == -1 ? (int)std::min<long long>(inner, 32) : 1;
  return s_outer == 1 ? (int)std::min<long long>(outer, 32) : 1;
}

cudaError_t launch_ring_mma(const RingParams& P, int sms, cudaStream_t s) {
  const int Co = P.kbound.x, Ci = P.kbound.y, KH = P.kbound.z, KW = P.kbound.w;
  RingMma R{};
  R.npos = P.outs / Co;
  R.K = (long long)Ci * KH * KW;
  const long long B = R.npos / ((long long)P.Ho * P.Wo);
  R.v_rows = run(P.Wo, P.v.s3, P.Ho == 1 ? B : 1, P.v.s0) >= run(KW, P.v.s3, KH == 1 ? Ci : 1, P.v.s1);
  R.w_rows = (P.w.s0 == 1 ? std::min(Co, 32) : 1) > run(KW, P.w.s3, KH == 1 ? Ci : 1, P.w.s1);
  const bool wide = P.t_mask >> 48;
  if (ring_tile(Co).rows == 64) return wide ? launch<8, 2, 2, 2>(P, R, sms, s) : launch<6, 2, 2, 2>(P, R, sms, s);
  if (ring_tile(Co).rows == 32) return wide ? launch<8, 1, 2, 2>(P, R, sms, s) : launch<6, 1, 2, 2>(P, R, sms, s);
  return wide ? launch<8, 1, 1, 4>(P, R, sms, s) : launch<6, 1, 1, 4>(P, R, sms, s);
}

}  // namespace pencil
