// Batched negacyclic NTT / INTT for one (polynomial, limb) per CTA.
//
// Sec. 5 ("NTT"): ring products in Z_q[X]/(X^N+1) become slot-wise after the
// transform.  Forward = Cooley-Tukey with twiddles psi^brv(m+i) (natural order
// in, bit-reversed evaluation order out); inverse = Gentleman-Sande with
// psi^-brv(m+i), then N^{-1}.  Harvey's lazy butterflies keep forward values
// in [0, 4q) and inverse values in [0, 2q); q < 2^62 keeps 4q < 2^64.  (The
// wider-range variants ct_bf8 / gs_bf4 of common.cuh measured slower on GB300
// with pencil_mul_probe and are not used here.)
//
// GB300 mapping: T = N / E threads each hold E = 2^LOGE coefficients in
// registers and run LOGE radix-2 stages between two shared-memory exchanges
// (a radix-2^LOGE round).  The first forward round reads its coefficients
// straight from the fused prologue (coalesced: thread t holds t + l*T); the
// result goes through shared memory once more so the fused epilogue sees pairs
// of consecutive slots (16-byte coalesced stores, one Philox block per pair).
#pragma once
#include <type_traits>
#include <utility>

#include <cooperative_groups.h>

#include "common.cuh"

namespace pencil {

// Final scaling of an inverse transform, applied by the engine (the mode's store
// receives the canonical scaled coefficient): N^{-1}, or N^{-1} qtil for
// decryption (the CRT factor folded in).
enum class InvScale { kNinv, kNqtil };

// Shared-memory slot of coefficient x: the low four index bits are XOR-ed with
// (bits 4..7) ^ (bits 5..8).  8-byte accesses are served per half-warp (16
// threads over the 16 bank pairs); with this swizzle every round's strided
// accesses and the epilogue's pair accesses hit 16 distinct bank pairs in each
// half-warp (two wavefronts per warp access, the minimum), for every N and radix.
template <int LOGN>
__device__ __forceinline__ int sidx(int x) {
  return x ^ (((x >> 4) ^ (x >> 5)) & 15);
}

template <int LOGN, int LOGE, int S0>
struct Round {
  static constexpr int K = (LOGN - S0) < LOGE ? (LOGN - S0) : LOGE;
  static constexpr int G = 1 << (LOGE - K);
  static constexpr int LOGD = LOGN - S0 - K;
  static constexpr int T = (1 << LOGN) >> LOGE;
  static constexpr int E = 1 << LOGE;

  static __device__ __forceinline__ int pos(int tau, int gg, int l) {
    int g = gg * T + tau;
    int B = g >> LOGD;
    int p = g & ((1 << LOGD) - 1);
    return (B << (LOGD + K)) + p + (l << LOGD);
  }
  static __device__ __forceinline__ void load(u64 (&v)[E], const u64* sm, int tau) {
#pragma unroll
    for (int gg = 0; gg < G; ++gg)
#pragma unroll
      for (int l = 0; l < (1 << K); ++l) v[gg * (1 << K) + l] = sm[sidx<LOGN>(pos(tau, gg, l))];
  }
  static __device__ __forceinline__ void store(const u64 (&v)[E], u64* sm, int tau) {
#pragma unroll
    for (int gg = 0; gg < G; ++gg)
#pragma unroll
      for (int l = 0; l < (1 << K); ++l) sm[sidx<LOGN>(pos(tau, gg, l))] = v[gg * (1 << K) + l];
  }
  // One radix-2 stage J of this round on every group the thread holds.
  template <int J, bool FWD>
  static __device__ __forceinline__ void stage(u64 (&v)[E], const ulonglong2* __restrict__ tw, int tau, u64 q,
                                               u64 q2) {
    constexpr int half = 1 << (K - 1 - J);
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
      const int B = (gg * T + tau) >> LOGD;
#pragma unroll
      for (int i = 0; i < (1 << J); ++i) {
        const ulonglong2 w = __ldg(tw + (1 << (S0 + J)) + (B << J) + i);
#pragma unroll
        for (int r = 0; r < half; ++r) {
          const int l = gg * (1 << K) + i * 2 * half + r;
          if constexpr (FWD)
            ct_butterfly(v[l], v[l + half], w.x, w.y, q, q2);
          else
            gs_butterfly(v[l], v[l + half], w.x, w.y, q, q2);
        }
      }
    }
  }
  template <int... J>
  static __device__ __forceinline__ void fwd_seq(std::integer_sequence<int, J...>, u64 (&v)[E],
                                                 const ulonglong2* tw, int tau, u64 q, u64 q2) {
    (stage<J, true>(v, tw, tau, q, q2), ...);
  }
  template <int... J>
  static __device__ __forceinline__ void inv_seq(std::integer_sequence<int, J...>, u64 (&v)[E],
                                                 const ulonglong2* tw, int tau, u64 q, u64 q2) {
    (stage<K - 1 - J, false>(v, tw, tau, q, q2), ...);
  }
  static __device__ __forceinline__ void fwd(u64 (&v)[E], const ulonglong2* __restrict__ tw, int tau, u64 q, u64 q2) {
    fwd_seq(std::make_integer_sequence<int, K>{}, v, tw, tau, q, q2);
  }
  static __device__ __forceinline__ void inv(u64 (&v)[E], const ulonglong2* __restrict__ tw, int tau, u64 q, u64 q2) {
    inv_seq(std::make_integer_sequence<int, K>{}, v, tw, tau, q, q2);
  }
};

// Forward rounds S0, S0 + LOGE, ...; on return the last round's values are in smem.
template <int LOGN, int LOGE, int S0>
struct FwdRounds {
  static __device__ __forceinline__ void run(u64 (&v)[1 << LOGE], u64* sm, const ulonglong2* tw, int tau, u64 q,
                                             u64 q2) {
    using R = Round<LOGN, LOGE, S0>;
    R::fwd(v, tw, tau, q, q2);
    if constexpr (S0 > 0) __syncthreads();  // previous round's readers are done
    R::store(v, sm, tau);
    __syncthreads();
    if constexpr (S0 + LOGE < LOGN) {
      Round<LOGN, LOGE, S0 + LOGE>::load(v, sm, tau);
      FwdRounds<LOGN, LOGE, S0 + LOGE>::run(v, sm, tw, tau, q, q2);
    }
  }
};

// Inverse rounds from S0 down to 0; on entry the values are in smem (synced);
// on return v holds the coefficients tau + l*T.
template <int LOGN, int LOGE, int S0>
struct InvRounds {
  static __device__ __forceinline__ void run(u64 (&v)[1 << LOGE], u64* sm, const ulonglong2* tw, int tau, u64 q,
                                             u64 q2) {
    using R = Round<LOGN, LOGE, S0>;
    R::load(v, sm, tau);
    R::inv(v, tw, tau, q, q2);
    if constexpr (S0 > 0) {
      __syncthreads();
      R::store(v, sm, tau);
      __syncthreads();
      InvRounds<LOGN, LOGE, S0 - LOGE>::run(v, sm, tw, tau, q, q2);
    }
  }
};

// Inverse modes that store few of their coefficients (Mode::occupied: whether any of the 32
// coefficients of a group is stored).
template <class M, class = void>
struct FewOutputs : std::false_type {};
template <class M>
struct FewOutputs<M, std::void_t<decltype(M::kFewOutputs)>> : std::bool_constant<M::kFewOutputs> {};

// Epilogue of an inverse transform: value(l) of coefficient tau + l T.  A warp's 32
// coefficients of one l are a group; where half of its groups or more store nothing they are
// skipped, each lane having looked up one of them.  (Other warps run the plain loop, whose
// loads the branches would serialise.)
template <class Mode, int N, int E, class Value>
__device__ __forceinline__ void store_inverse(const DevCtx& ctx, const typename Mode::Params& P, const LimbConst& lc,
                                              int poly, int limb, int tau, Value value) {
  constexpr int T = N / E;
  if constexpr (FewOutputs<Mode>::value) {
    const int lane = tau & 31;
    const u32 some =
        __ballot_sync(0xffffffffu, lane < E && Mode::occupied(P, (tau >> 5) + (lane < E ? lane : 0) * (T / 32)));
    if (2 * __popc(some) <= E) {
#pragma unroll
      for (int l = 0; l < E; ++l)
        if (some >> l & 1u) Mode::template store<N>(ctx, P, lc, poly, limb, tau + l * T, value(l));
      return;
    }
  }
#pragma unroll
  for (int l = 0; l < E; ++l) Mode::template store<N>(ctx, P, lc, poly, limb, tau + l * T, value(l));
}

template <int LOGN, int LOGE_>
struct NttCfg {
  static constexpr int LOGE = LOGE_;
  static constexpr int N = 1 << LOGN;
  static constexpr int E = 1 << LOGE;
  static constexpr int T = N >> LOGE;
  static constexpr int LAST_S0 = ((LOGN - 1) / LOGE) * LOGE;
  static constexpr size_t SMEM = (size_t)N * sizeof(u64);
  // two CTAs (two transforms) per SM when their threads and shared memory fit
  static constexpr int MIN_BLOCKS = (T <= 512 && 2 * SMEM <= 227 * 1024) ? 2 : 1;
};

// Forward transform of (poly, limb) with a fused prologue (Mode::load,
// canonical coefficient e) and epilogue (Mode::store2, canonical slots e, e + 1).
template <int LOGN, int LOGE, class Mode>
__device__ __forceinline__ void ntt_fwd_run(const DevCtx& ctx, const typename Mode::Params& P, int poly, int limb,
                                            u64* sm) {
  using C = NttCfg<LOGN, LOGE>;
  const int tau = threadIdx.x;
  const LimbConst& lc = ctx.limb[limb];
  const typename Mode::Pre pre(ctx, P, poly);
  const u64 q = lc.q, q2 = 2 * q;
  const ulonglong2* tw = ctx.tw_fwd + (size_t)limb * C::N;
  u64 v[C::E];
  if constexpr (Mode::kHeavyLoad) {
    // Long prologue (gathers, multiplies): a loop through shared memory bounds
    // the code size (kLoadUnroll iterations in flight); each thread re-reads
    // only the slots it wrote.
#pragma unroll(Mode::kLoadUnroll)
    for (int l = 0; l < C::E; ++l) {
      const int e = tau + l * C::T;
      sm[sidx<LOGN>(e)] = Mode::template load<C::N, false>(ctx, P, pre, lc, poly, limb, e);
    }
#pragma unroll
    for (int l = 0; l < C::E; ++l) v[l] = sm[sidx<LOGN>(tau + l * C::T)];
    __syncthreads();
  } else {
#pragma unroll
    for (int l = 0; l < C::E; ++l) v[l] = Mode::template load<C::N, false>(ctx, P, pre, lc, poly, limb, tau + l * C::T);
  }
  FwdRounds<LOGN, C::LOGE, 0>::run(v, sm, tw, tau, q, q2);
  if constexpr (Mode::kQuad) {
#pragma unroll(Mode::kEpilogueUnroll)
    for (int l = 0; l < C::E / 4; ++l) {
      const int e = 4 * (tau + l * C::T);
      u64 x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = canon4(sm[sidx<LOGN>(e + i)], q, q2);
      Mode::template store4<C::N, false>(ctx, P, lc, poly, limb, e, x);
    }
  } else {
#pragma unroll(Mode::kEpilogueUnroll)
    for (int l = 0; l < C::E / 2; ++l) {
      const int e = 2 * (tau + l * C::T);
      const u64 x0 = canon4(sm[sidx<LOGN>(e)], q, q2);
      const u64 x1 = canon4(sm[sidx<LOGN>(e + 1)], q, q2);
      Mode::template store2<C::N, false>(ctx, P, lc, poly, limb, e, x0, x1);
    }
  }
}

// Inverse transform of (poly, limb) with a fused prologue (Mode::load, value in
// [0, 2q)) and epilogue (Mode::store, canonical coefficient e).
template <int LOGN, int LOGE, class Mode>
__device__ __forceinline__ void ntt_inv_run(const DevCtx& ctx, const typename Mode::Params& P, int poly, int limb,
                                            u64* sm) {
  using C = NttCfg<LOGN, LOGE>;
  const int tau = threadIdx.x;
  const LimbConst& lc = ctx.limb[limb];
  const typename Mode::Pre pre(ctx, P, poly);
  const u64 q = lc.q, q2 = 2 * q;
  const ulonglong2* tw = ctx.tw_inv + (size_t)limb * C::N;
  u64 v[C::E];
#pragma unroll(Mode::kLoadUnroll)
  for (int l = 0; l < C::E; ++l) {
    const int e = tau + l * C::T;
    sm[sidx<LOGN>(e)] = Mode::template load<C::N, false>(ctx, P, pre, lc, poly, limb, e);
  }
  __syncthreads();
  InvRounds<LOGN, C::LOGE, C::LAST_S0>::run(v, sm, tw, tau, q, q2);
  // v in [0, 2q); scaled here by the mode's kappa (N^{-1}, possibly with its own constant folded in)
  const bool ninv = Mode::kInvScale == InvScale::kNinv;
  const u64 kap = ninv ? lc.ninv : lc.nqtil, kaps = ninv ? lc.ninvs : lc.nqtils;
  store_inverse<Mode, C::N, C::E>(ctx, P, lc, poly, limb, tau, [&](int l) { return mul_shoup(v[l], kap, kaps, q); });
}

// ------------------------------------------------------------------ pseudo-Mersenne engine
// The same transforms for primes q = 2^b - c with signed split products (mul_split,
// common.cuh): no correction step inside a butterfly and no added multiple of q;
// signed values grow lazily and are folded only where the bound requires it
// (units of 2^b):
//  * forward: from [0, 1], k = 1 .. 4 stages stay inside -(1.65, 3.33, 5.06, 6.96) ..
//    (2.65, 4.33, 6.06, 7.96) for primes of every length, so the registers are folded once per round of at most
//    four stages (rounds of five fold after their second stage too); before the last
//    fold 4 q (at most two stages) or 8 q is added, so that it is unsigned and one
//    conditional subtraction is canonical;
//  * inverse: a stage doubles the range of its sums, so the sums of every second
//    stage (counted from the first inverse stage) are folded; the last stage's
//    products (its scaling) start from 2 q, which makes them positive.
// Shared memory holds the N words with two spare words after every 32
// (slot ph(x)): every round's accesses are conflict-free and a thread's words of
// one round sit at compile-time offsets from one base address.  The last
// forward round of at most 2 stages runs inside the epilogue on groups of 2 or 4
// consecutive slots read from shared memory, and the first inverse round of at
// most 2 stages inside the prologue, which saves a shared-memory round trip
// (N = 8192 with radix 2^4: rounds of 4, 4, 4 and 1 stages).

__device__ __forceinline__ constexpr int ph(int x) { return x + 2 * (x >> 5); }

template <int LOGN, int LOGE>
struct FCfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int E = 1 << LOGE;
  static constexpr int T = N >> LOGE;
  static constexpr int R = (LOGN + LOGE - 1) / LOGE;    // rounds
  static constexpr int SL = (R - 1) * LOGE;              // first stage of the last round
  static constexpr int KL = LOGN - SL;                   // its stages, 1 .. LOGE
  static constexpr bool FUSE = KL <= 2;
  static constexpr size_t SMEM = (size_t)(N + 2 * (N >> 5)) * sizeof(u64);
  static constexpr int MIN_BLOCKS = (T <= 512 && 2 * SMEM <= 227 * 1024) ? 2 : 1;
};

// Barrier between two shared-memory phases: the warp's own when every slot the
// following phase touches was last touched by the same warp, the CTA's otherwise.
template <bool WARP_LOCAL>
__device__ __forceinline__ void phase_sync() {
  if constexpr (WARP_LOCAL)
    __syncwarp();
  else
    __syncthreads();
}

// Round S0 of the fold engine: K stages on G groups of 2^K words per thread;
// group gg of thread tau is at positions base + l 2^LOGD, slot ph(base) + ph(l 2^LOGD).
// A round is warp-local (kLocal) when warp w reads and writes only the 32 E
// consecutive positions [32 E w, 32 E (w + 1)): full rounds with LOGD <= 5, and
// the last (partial) round, whose G groups per thread are numbered warp by warp
// (group 32 G w + 32 gg + lane) for that purpose.  Between two warp-local phases
// the exchange through shared memory needs only __syncwarp.
template <int LOGN, int LOGE, int S0>
struct FRound {
  static constexpr int K = (LOGN - S0) < LOGE ? (LOGN - S0) : LOGE;
  static constexpr int G = 1 << (LOGE - K);
  static constexpr int LOGD = LOGN - S0 - K;
  static constexpr int T = (1 << LOGN) >> LOGE;
  static constexpr int E = 1 << LOGE;
  static constexpr bool kLocal = (K < LOGE) || (LOGD <= 5);
  static_assert(T % 32 == 0, "whole warps");
  static_assert(K == LOGE || LOGD == 0, "only the last round is partial");

  static __device__ __forceinline__ int grp(int tau, int gg) {
    if constexpr (G == 1)
      return tau;
    else
      return ((tau >> 5) << (5 + LOGE - K)) + (gg << 5) + (tau & 31);
  }
  static __device__ __forceinline__ int base(int tau, int gg) {
    const int g = grp(tau, gg);
    return ph(((g >> LOGD) << (LOGD + K)) + (g & ((1 << LOGD) - 1)));
  }
  static __device__ __forceinline__ void load(u64 (&v)[E], const u64* sm, int tau) {
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
      const u64* b = sm + base(tau, gg);
#pragma unroll
      for (int l = 0; l < (1 << K); ++l) v[gg * (1 << K) + l] = b[ph(l << LOGD)];
    }
  }
  static __device__ __forceinline__ void store(const u64 (&v)[E], u64* sm, int tau) {
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
      u64* b = sm + base(tau, gg);
#pragma unroll
      for (int l = 0; l < (1 << K); ++l) b[ph(l << LOGD)] = v[gg * (1 << K) + l];
    }
  }
  // Stage J of the round (global stage S0 + J), forward.
  template <int J>
  static __device__ __forceinline__ void fwd_stage(u64 (&v)[E], const uint4* __restrict__ tw, int tau, const FoldC& f, int root) {
    constexpr int half = 1 << (K - 1 - J);
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
      const int B = grp(tau, gg) >> LOGD;
#pragma unroll
      for (int i = 0; i < (1 << J); ++i) {
        const uint4 w = __ldg(tw + (root << (S0 + J)) + (B << J) + i);
#pragma unroll
        for (int r = 0; r < half; ++r) {
          const int l = gg * (1 << K) + i * 2 * half + r;
          ct_split(v[l], v[l + half], w, f);
        }
      }
    }
    if constexpr (K == 5 && J == 1) {   // five stages from [0, 1] would leave 64 bits
#pragma unroll
      for (int l = 0; l < E; ++l) v[l] = fold_s(v[l], f);
    }
  }
  // Stage J of the round, inverse; the stages at odd positions of the inverse order
  // (LOGN - 1 - (S0 + J)) fold their sums.
  template <int J>
  static __device__ __forceinline__ void inv_stage(u64 (&v)[E], const uint4* __restrict__ tw, int tau, const FoldC& f, int root) {
    constexpr int half = 1 << (K - 1 - J);
    constexpr bool odd = ((LOGN - 1 - (S0 + J)) & 1) != 0;
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
      const int B = grp(tau, gg) >> LOGD;
#pragma unroll
      for (int i = 0; i < (1 << J); ++i) {
        const uint4 w = __ldg(tw + (root << (S0 + J)) + (B << J) + i);
#pragma unroll
        for (int r = 0; r < half; ++r) {
          const int l = gg * (1 << K) + i * 2 * half + r;
          gs_split(v[l], v[l + half], w, f);
          if constexpr (odd) v[l] = fold_s(v[l], f);
        }
      }
    }
  }
  template <int... J>
  static __device__ __forceinline__ void fwd_seq(std::integer_sequence<int, J...>, u64 (&v)[E],
                                                 const uint4* tw, int tau, const FoldC& f, int root) {
    (fwd_stage<J>(v, tw, tau, f, root), ...);
  }
  // Round 0 of the inverse with the transform's final scaling kappa merged into
  // its last stage (global stage 0, whose butterflies all use w1 = tw[1]):
  //   x' = (x + y) kappa + 2 q,  y' = (x - y) (w1 kappa) + 2 q,  both in (0.9 q, 4.1 q),
  // N / 2 products instead of the stage's N / 2 and the N of a separate scaling.
  // sc = split twiddles {kappa, w1 kappa}.
  static __device__ __forceinline__ void inv_scaled(u64 (&v)[E], const uint4* tw, int tau, const FoldC& f, u64 q2,
                                                    const uint4* sc) {
    static_assert(S0 == 0 && G == 1 && K == LOGE, "the first round, full");
    inv_seq(std::make_integer_sequence<int, K - 1>{}, v, tw, tau, f, 1);
    const uint4 k = sc[0], wk = sc[1];
#pragma unroll
    for (int r = 0; r < E / 2; ++r) {
      const u64 x = v[r], y = v[r + E / 2];
      v[r] = mul_split(q2, x + y, k, f);
      v[r + E / 2] = mul_split(q2, x - y, wk, f);
    }
  }
  // Stages K - 1 .. 0 (inverse order), or K - 1 .. 1 with sizeof...(J) = K - 1.
  template <int... J>
  static __device__ __forceinline__ void inv_seq(std::integer_sequence<int, J...>, u64 (&v)[E],
                                                 const uint4* tw, int tau, const FoldC& f, int root) {
    (inv_stage<K - 1 - J>(v, tw, tau, f, root), ...);
  }
  static __device__ __forceinline__ void fwd(u64 (&v)[E], const uint4* tw, int tau, const FoldC& f, int root) {
    fwd_seq(std::make_integer_sequence<int, K>{}, v, tw, tau, f, root);
  }
  // Stages j0 .. K - 1 only (j0 uniform across the CTA).
  template <int... J>
  static __device__ __forceinline__ void fwd_from_seq(std::integer_sequence<int, J...>, int j0, u64 (&v)[E],
                                                      const uint4* tw, int tau, const FoldC& f, int root) {
    ((J >= j0 ? fwd_stage<J>(v, tw, tau, f, root) : void()), ...);
  }
  static __device__ __forceinline__ void fwd_from(int j0, u64 (&v)[E], const uint4* tw, int tau, const FoldC& f, int root) {
    fwd_from_seq(std::make_integer_sequence<int, K>{}, j0, v, tw, tau, f, root);
  }
  static __device__ __forceinline__ void inv(u64 (&v)[E], const uint4* tw, int tau, const FoldC& f, int root) {
    inv_seq(std::make_integer_sequence<int, K>{}, v, tw, tau, f, root);
  }
};

// Full forward rounds S0, S0 + LOGE, ... before the last round; round 0 takes its
// words from registers (the prologue's coefficients tau + l T), the others from
// shared memory.  Each round folds its words and leaves them in shared memory.
template <int LOGN, int LOGE, int S0>
struct FFwdRounds {
  static __device__ __forceinline__ void run(u64 (&v)[1 << LOGE], u64* sm, const uint4* tw, int tau, const FoldC& f, int root) {
    using Rd = FRound<LOGN, LOGE, S0>;
    if constexpr (S0 > 0) Rd::load(v, sm, tau);
    Rd::fwd(v, tw, tau, f, root);
#pragma unroll
    for (int l = 0; l < (1 << LOGE); ++l) v[l] = fold_s(v[l], f);
    if constexpr (S0 > 0) phase_sync<Rd::kLocal>();   // every reader of these slots is done
    Rd::store(v, sm, tau);
    phase_sync<Rd::kLocal>();   // the following rounds are warp-local once this one is
    if constexpr (S0 + LOGE < FCfg<LOGN, LOGE>::SL) FFwdRounds<LOGN, LOGE, S0 + LOGE>::run(v, sm, tw, tau, f, root);
  }
};

// Inverse rounds from S0 down to 0 (words in shared memory on entry, synced); on
// return v holds the coefficients tau + l T.
template <int LOGN, int LOGE, int S0, bool SCALED = true>
struct FInvRounds {
  static __device__ __forceinline__ void run(u64 (&v)[1 << LOGE], u64* sm, const uint4* tw, int tau, const FoldC& f,
                                             u64 q2, const uint4* sc, int root) {
    using Rd = FRound<LOGN, LOGE, S0>;
    Rd::load(v, sm, tau);
    if constexpr (S0 == 0 && SCALED)
      Rd::inv_scaled(v, tw, tau, f, q2, sc);
    else
      Rd::inv(v, tw, tau, f, root);
    if constexpr (S0 > 0) {
      phase_sync<Rd::kLocal>();
      Rd::store(v, sm, tau);
      phase_sync<Rd::kLocal && FRound<LOGN, LOGE, S0 - LOGE>::kLocal>();
      FInvRounds<LOGN, LOGE, S0 - LOGE, SCALED>::run(v, sm, tw, tau, f, q2, sc, root);
    }
  }
};

// The last forward round's KL stages on one group of W = 2^KL consecutive slots
// (group index g: positions g W .. g W + W - 1), then canonical values.
template <int LOGN, int LOGE>
__device__ __forceinline__ void fold_last_fwd(u64* u, const uint4* __restrict__ tw, int g, const FoldC& f, u64 q,
                                              u64 off, int root) {
  using C = FCfg<LOGN, LOGE>;
  constexpr int W = 1 << C::KL;
#pragma unroll
  for (int J = 0; J < C::KL; ++J) {
    const int half = W >> (J + 1);
#pragma unroll
    for (int i = 0; i < (1 << J); ++i) {
      const uint4 w = __ldg(tw + (root << (C::SL + J)) + (g << J) + i);
#pragma unroll
      for (int r = 0; r < half; ++r) ct_split(u[i * 2 * half + r], u[i * 2 * half + r + half], w, f);
    }
  }
#pragma unroll
  for (int i = 0; i < W; ++i) u[i] = csub(fold_u(u[i] + off, f), q);
}

// The first inverse round's KL stages (inverse steps 0 .. KL - 1) on one group.
template <int LOGN, int LOGE>
__device__ __forceinline__ void fold_first_inv(u64 (&u)[1 << FCfg<LOGN, LOGE>::KL],
                                               const uint4* __restrict__ tw, int g, const FoldC& f, int root) {
  using C = FCfg<LOGN, LOGE>;
  constexpr int W = 1 << C::KL;
#pragma unroll
  for (int J = C::KL - 1; J >= 0; --J) {
    const int half = W >> (J + 1);
    const bool odd = ((LOGN - 1 - (C::SL + J)) & 1) != 0;
#pragma unroll
    for (int i = 0; i < (1 << J); ++i) {
      const uint4 w = __ldg(tw + (root << (C::SL + J)) + (g << J) + i);
#pragma unroll
      for (int r = 0; r < half; ++r) {
        u64& x = u[i * 2 * half + r];
        gs_split(x, u[i * 2 * half + r + half], w, f);
        if (odd) x = fold_s(x, f);
      }
    }
  }
}

// Modes whose input polynomials may have a short support (Mode::support(P):
// coefficients from there on are zero).
template <class M, class = void>
struct SparseInput : std::false_type {};
template <class M>
struct SparseInput<M, std::void_t<decltype(M::kSparse)>> : std::bool_constant<M::kSparse> {};

// Modes some of whose polynomials are contiguous words (Mode::direct, or null).
template <class M, class = void>
struct DirectInput : std::false_type {};
template <class M>
struct DirectInput<M, std::void_t<decltype(M::kDirect)>> : std::bool_constant<M::kDirect> {};

// Forward rounds 0 and 1 of a polynomial of degree < sup <= T.  After s
// Cooley-Tukey stages, block b of N / 2^s words holds p mod (X^{N/2^s} - zeta_b),
// which is p itself while deg p < N / 2^s: the first LOGN - ceil(log2 sup)
// stages only copy.  Round 0 (LOGE stages) is therefore skipped whole, and so
// are the first j stages of round 1 where sup <= T / 2^j; round 1 then starts
// from word x = p[x mod (N / 2^(LOGE + j))], read from the T prologue values in
// shared memory (one gather per thread instead of E).  The values are those the
// skipped butterflies leave (ct_split(a, 0) = (a, a)).  Leaves round 1's words, folded, in shared memory.
template <int LOGN, int LOGE, class Mode>
__device__ __forceinline__ void fold_sparse_head(const DevCtx& ctx, const typename Mode::Params& P,
                                                 const typename Mode::Pre& pre, const LimbConst& lc, int poly, int limb, int sup,
                                                 u64 (&v)[1 << LOGE],
                                                 u64* sm, const uint4* tw, int tau, const FoldC& f) {
  using C = FCfg<LOGN, LOGE>;
  using R1 = FRound<LOGN, LOGE, LOGE>;
  static_assert(R1::K == LOGE && R1::G == 1, "round 1 must be a full round");
  sm[ph(tau)] = tau < sup ? Mode::template load<C::N, true>(ctx, P, pre, lc, poly, limb, tau) : 0ull;
  int j = 0;
  while (j < LOGE && sup <= (C::T >> (j + 1))) ++j;
  __syncthreads();
  constexpr int D1 = 1 << R1::LOGD;   // round 1: thread tau holds words base + l D1
  const int m = (C::E >> j) - 1;
  const u64* b = sm + ph(tau & (D1 - 1));
#pragma unroll
  for (int l = 0; l < C::E; ++l) v[l] = b[ph(D1 * (l & m))];
  R1::fwd_from(j, v, tw, tau, f, 1);
#pragma unroll
  for (int l = 0; l < C::E; ++l) v[l] = fold_s(v[l], f);
  __syncthreads();   // every thread has read the prologue values
  R1::store(v, sm, tau);
  phase_sync<R1::kLocal>();
  if constexpr (2 * LOGE < C::SL) FFwdRounds<LOGN, LOGE, 2 * LOGE>::run(v, sm, tw, tau, f, 1);
}

// Last round and epilogue of a (sub)transform of 2^LOGN words whose slots are e0, e0 + 1,
// ... of a polynomial of 2^LOGP.
template <int LOGN, int LOGE, int LOGP, class Mode>
__device__ __forceinline__ void fold_tail(const DevCtx& ctx, const typename Mode::Params& P, const LimbConst& lc,
                                          int poly, int limb, u64 (&v)[1 << LOGE], u64* sm, const uint4* tw, int tau,
                                          const FoldC& f, int root, int e0) {
  using C = FCfg<LOGN, LOGE>;
  constexpr int NFULL = 1 << LOGP;
  const u64 q = lc.q;
  if constexpr (C::FUSE) {
    // groups of GW consecutive slots per iteration: the last round's groups of
    // W = 2^KL, gathered in fours for modes that store four coefficients at a time
    constexpr int W = 1 << C::KL;
    constexpr int GW = (Mode::kQuad && W < 4) ? 4 : W;
    // group k = 32 (E / GW) w + 32 j + lane: warp w's own positions [32 E w, 32 E (w + 1))
    const int kbase = (tau >> 5) * (32 * C::E / GW) + (tau & 31);
#pragma unroll(Mode::kEpilogueUnroll)
    for (int j = 0; j < C::E / GW; ++j) {
      const int k = kbase + 32 * j;
      u64 u[GW];
      const ulonglong2* b = reinterpret_cast<const ulonglong2*>(sm + ph(k * GW));
#pragma unroll
      for (int i = 0; i < GW / 2; ++i) {
        const ulonglong2 x = b[i];
        u[2 * i] = x.x;
        u[2 * i + 1] = x.y;
      }
#pragma unroll
      for (int s = 0; s < GW / W; ++s) fold_last_fwd<LOGN, LOGE>(u + s * W, tw, k * (GW / W) + s, f, q, 4 * q, root);
      if constexpr (Mode::kQuad) {
#pragma unroll
        for (int i = 0; i < GW / 4; ++i) Mode::template store4<NFULL, true>(ctx, P, lc, poly, limb, e0 + k * GW + 4 * i, u + 4 * i);
      } else {
#pragma unroll
        for (int i = 0; i < GW / 2; ++i)
          Mode::template store2<NFULL, true>(ctx, P, lc, poly, limb, e0 + k * GW + 2 * i, u[2 * i], u[2 * i + 1]);
      }
    }
  } else {
    using Rd = FRound<LOGN, LOGE, C::SL>;
    Rd::load(v, sm, tau);
    Rd::fwd(v, tw, tau, f, root);
#pragma unroll
    for (int l = 0; l < C::E; ++l) v[l] = csub(fold_u(v[l] + 8 * q, f), q);
    static_assert(Rd::kLocal, "the last round is warp-local");
    __syncwarp();
    Rd::store(v, sm, tau);
    __syncwarp();
    // the epilogue's groups are warp w's own positions [32 E w, 32 E (w + 1))
    const int wbase = (tau >> 5) * 32 * C::E, lane = tau & 31;
    if constexpr (Mode::kQuad) {
#pragma unroll(Mode::kEpilogueUnroll)
      for (int l = 0; l < C::E / 4; ++l) {
        const int e = wbase + 4 * (lane + 32 * l);
        const ulonglong2* b = reinterpret_cast<const ulonglong2*>(sm + ph(e));
        const ulonglong2 x01 = b[0], x23 = b[1];
        u64 x[4] = {x01.x, x01.y, x23.x, x23.y};
        Mode::template store4<NFULL, true>(ctx, P, lc, poly, limb, e0 + e, x);
      }
    } else {
#pragma unroll(Mode::kEpilogueUnroll)
      for (int l = 0; l < C::E / 2; ++l) {
        const int e = wbase + 2 * (lane + 32 * l);
        const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(sm + ph(e));
        Mode::template store2<NFULL, true>(ctx, P, lc, poly, limb, e0 + e, x.x, x.y);
      }
    }
  }
}

template <int LOGN, int LOGE, class Mode>
__device__ __forceinline__ void ntt_fwd_run_fold(const DevCtx& ctx, const typename Mode::Params& P, int poly,
                                                 int limb, u64* sm) {
  using C = FCfg<LOGN, LOGE>;
  const int tau = threadIdx.x;
  const LimbConst& lc = ctx.limb[limb];
  const typename Mode::Pre pre(ctx, P, poly);
  const FoldC f(lc);
  const uint4* tw = ctx.tw_fwd_f + (size_t)limb * C::N;
  u64 v[C::E];
  bool dense = true;
  if constexpr (SparseInput<Mode>::value && C::R >= 3) {
    const int sup = Mode::support(P);
    if (sup <= C::T) {
      dense = false;
      fold_sparse_head<LOGN, LOGE, Mode>(ctx, P, pre, lc, poly, limb, sup, v, sm, tw, tau, f);
    }
  }
  if (dense) {
    const u64* src = nullptr;
    if constexpr (DirectInput<Mode>::value) src = Mode::template direct<C::N>(P, poly);
    if (src) {   // a contiguous polynomial
      if constexpr (DirectInput<Mode>::value) {
        if (!Mode::noisy(ctx)) {   // all the thread's words in flight at once
#pragma unroll
          for (int l = 0; l < C::E; ++l) v[l] = __ldg(src + tau + l * C::T);
#pragma unroll
          for (int l = 0; l < C::E; ++l) v[l] = Mode::direct_value(ctx, v[l], 0, lc, f);
        } else {   // one Philox block per four consecutive words
#pragma unroll 1
          for (int j = 0; j < C::E / 4; ++j) {
            const int e = 4 * (tau + j * C::T);
            const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(src + e));
            const ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2*>(src + e) + 1);
            const Philox4 w = Mode::noise(P, poly, e);
            sm[ph(e)] = Mode::direct_value(ctx, a.x, Mode::noise_add(ctx, w.v[0]), lc, f);
            sm[ph(e + 1)] = Mode::direct_value(ctx, a.y, Mode::noise_add(ctx, w.v[1]), lc, f);
            sm[ph(e + 2)] = Mode::direct_value(ctx, b.x, Mode::noise_add(ctx, w.v[2]), lc, f);
            sm[ph(e + 3)] = Mode::direct_value(ctx, b.y, Mode::noise_add(ctx, w.v[3]), lc, f);
          }
          __syncthreads();
#pragma unroll
          for (int l = 0; l < C::E; ++l) v[l] = sm[ph(tau + l * C::T)];
        }
      }
    } else if constexpr (Mode::kHeavyLoad) {
#pragma unroll(Mode::kLoadUnroll)
      for (int l = 0; l < C::E; ++l) {
        const int e = tau + l * C::T;
        sm[ph(e)] = Mode::template load<C::N, true>(ctx, P, pre, lc, poly, limb, e);
      }
#pragma unroll
      for (int l = 0; l < C::E; ++l) v[l] = sm[ph(tau + l * C::T)];
    } else {
#pragma unroll
      for (int l = 0; l < C::E; ++l) v[l] = Mode::template load<C::N, true>(ctx, P, pre, lc, poly, limb, tau + l * C::T);
    }
    // (round 0 stores each thread's words at the slots it read them from: no barrier needed here)
    FFwdRounds<LOGN, LOGE, 0>::run(v, sm, tw, tau, f, 1);
  }
  fold_tail<LOGN, LOGE, LOGN, Mode>(ctx, P, lc, poly, limb, v, sm, tw, tau, f, 1, 0);
}

// Prologue and rounds of an inverse (sub)transform of 2^LOGN words (slots e0, e0 + 1, ...
// of a polynomial of 2^LOGP); on return v holds the coefficients tau + l T.
template <int LOGN, int LOGE, int LOGP, class Mode, bool SCALED>
__device__ __forceinline__ void fold_inv_rounds(const DevCtx& ctx, const typename Mode::Params& P,
                                                const typename Mode::Pre& pre, const LimbConst& lc, int poly, int limb,
                                                u64 (&v)[1 << LOGE], u64* sm, const uint4* tw, int tau, const FoldC& f,
                                                u64 q2, const uint4* sc, int root, int e0) {
  using C = FCfg<LOGN, LOGE>;
  constexpr int NFULL = 1 << LOGP;
  if constexpr (C::FUSE) {
    constexpr int W = 1 << C::KL;
    // group g = 32 (E / W) w + 32 j + lane: warp w's own positions [32 E w, 32 E (w + 1))
    const int gbase = (tau >> 5) * (32 * C::E / W) + (tau & 31);
#pragma unroll(Mode::kLoadUnroll)
    for (int j = 0; j < (C::E >> C::KL); ++j) {
      const int g = gbase + 32 * j;
      u64 u[W];
#pragma unroll
      for (int i = 0; i < W; i += 2)
        Mode::template load2<NFULL>(ctx, P, lc, poly, limb, e0 + g * W + i, u[i], u[i + 1]);
      fold_first_inv<LOGN, LOGE>(u, tw, g, f, root);
      ulonglong2* b = reinterpret_cast<ulonglong2*>(sm + ph(g * W));
#pragma unroll
      for (int i = 0; i < W / 2; ++i) b[i] = make_ulonglong2(u[2 * i], u[2 * i + 1]);
    }
    if constexpr (C::SL > 0) {
      phase_sync<FRound<LOGN, LOGE, C::SL - LOGE>::kLocal>();
      FInvRounds<LOGN, LOGE, C::SL - LOGE, SCALED>::run(v, sm, tw, tau, f, q2, sc, root);
    } else {
      __syncthreads();
    }
  } else {
    // warp w loads its own positions [32 E w, 32 E (w + 1)), which the first
    // (warp-local) inverse round reads
    const int wbase = (tau >> 5) * 32 * C::E + (tau & 31);
#pragma unroll(Mode::kLoadUnroll)
    for (int l = 0; l < C::E; ++l) {
      const int e = wbase + 32 * l;
      sm[ph(e)] = Mode::template load<NFULL, true>(ctx, P, pre, lc, poly, limb, e0 + e);
    }
    static_assert(FRound<LOGN, LOGE, C::SL>::kLocal, "the last round is warp-local");
    __syncwarp();
    FInvRounds<LOGN, LOGE, C::SL, SCALED>::run(v, sm, tw, tau, f, q2, sc, root);
  }
}

template <int LOGN, int LOGE, class Mode>
__device__ __forceinline__ void ntt_inv_run_fold(const DevCtx& ctx, const typename Mode::Params& P, int poly,
                                                 int limb, u64* sm) {
  using C = FCfg<LOGN, LOGE>;
  const int tau = threadIdx.x;
  const LimbConst& lc = ctx.limb[limb];
  const typename Mode::Pre pre(ctx, P, poly);
  const u64 q = lc.q;
  const FoldC f(lc);
  const uint4* tw = ctx.tw_inv_f + (size_t)limb * C::N;
  const uint4* sc = Mode::kInvScale == InvScale::kNinv ? lc.sc_ninv : lc.sc_nqtil;
  u64 v[C::E];
  fold_inv_rounds<LOGN, LOGE, LOGN, Mode, true>(ctx, P, pre, lc, poly, limb, v, sm, tw, tau, f, 2 * q, sc, 1, 0);
  // v in (0.9 q, 4.1 q), already scaled by the mode's kappa in the last stage
  store_inverse<Mode, C::N, C::E>(ctx, P, lc, poly, limb, tau, [&](int l) { return csub(fold_u(v[l], f), q); });
}

// One transform on a cluster of four CTAs, for launches too small to fill the GPU: after
// two Cooley-Tukey stages block r of N / 4 words is a transform of its own, with the
// twiddles of the subtree under node 4 + r.  CTA r evaluates the prologue of the r-th
// quarter of the coefficients into its shared memory, combines the four quarters for its
// block (three products a word, reading the others' through distributed shared memory)
// and transforms the block alone; the inverse runs its block's stages first and then the
// last two on a quarter of the block positions.  Radix 2^3: N / 32 threads a CTA, so a
// lone transform runs on 4 SMs with a quarter of the words each.
template <int LOGN>
struct Quad {
  static constexpr int LOGM = LOGN - 2, LOGE = 3, M = 1 << LOGM;
  using C = FCfg<LOGM, LOGE>;
};

template <int LOGN, class Mode>
__device__ __forceinline__ void quad_fwd(const DevCtx& ctx, const typename Mode::Params& P, int poly, int limb,
                                         u64* sm) {
  namespace cg = cooperative_groups;
  using Q = Quad<LOGN>;
  using C = typename Q::C;
  cg::cluster_group cl = cg::this_cluster();
  const int tau = threadIdx.x, rank = (int)cl.block_rank(), root = 4 + rank;
  const LimbConst& lc = ctx.limb[limb];
  const typename Mode::Pre pre(ctx, P, poly);
  const FoldC f(lc);
  const uint4* tw = ctx.tw_fwd_f + (size_t)limb * (1 << LOGN);
  u64 v[C::E];
  bool copied = false;
  if constexpr (SparseInput<Mode>::value) {
    const int sup = Mode::support(P);
    if (sup <= Q::M) {   // the first two stages only copy: every block starts from the same words
      copied = true;
#pragma unroll
      for (int l = 0; l < C::E; ++l) {
        const int p = tau + l * C::T;
        v[l] = p < sup ? Mode::template load<1 << LOGN, true>(ctx, P, pre, lc, poly, limb, p) : 0ull;
      }
    }
  }
  if (!copied) {
#pragma unroll
    for (int l = 0; l < C::E; ++l) {
      const int p = tau + l * C::T;
      sm[ph(p)] = Mode::template load<1 << LOGN, true>(ctx, P, pre, lc, poly, limb, rank * Q::M + p);
    }
    const uint4 w1 = __ldg(tw + 1), w2 = __ldg(tw + 2 + (rank >> 1));
    const u64* x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = cl.map_shared_rank(sm, k);
    cl.sync();
#pragma unroll
    for (int l = 0; l < C::E; ++l) {
      const int at = ph(tau + l * C::T);
      const u64 a = mul_split(0, x[2][at], w1, f), b = mul_split(0, x[3][at], w1, f);
      const u64 c = rank & 2 ? x[0][at] - a : x[0][at] + a, d = rank & 2 ? x[1][at] - b : x[1][at] + b;
      const u64 t = mul_split(0, d, w2, f);
      v[l] = fold_s(rank & 1 ? c - t : c + t, f);
    }
    cl.sync();   // every quarter has been read: the rounds may write shared memory
  }
  FFwdRounds<Q::LOGM, Q::LOGE, 0>::run(v, sm, tw, tau, f, root);
  fold_tail<Q::LOGM, Q::LOGE, LOGN, Mode>(ctx, P, lc, poly, limb, v, sm, tw, tau, f, root, rank * Q::M);
}

template <int LOGN, class Mode>
__device__ __forceinline__ void quad_inv(const DevCtx& ctx, const typename Mode::Params& P, int poly, int limb,
                                         u64* sm) {
  namespace cg = cooperative_groups;
  using Q = Quad<LOGN>;
  using C = typename Q::C;
  cg::cluster_group cl = cg::this_cluster();
  const int tau = threadIdx.x, rank = (int)cl.block_rank(), root = 4 + rank;
  const LimbConst& lc = ctx.limb[limb];
  const typename Mode::Pre pre(ctx, P, poly);
  const u64 q = lc.q;
  const FoldC f(lc);
  const uint4* tw = ctx.tw_inv_f + (size_t)limb * (1 << LOGN);
  const uint4* sc = Mode::kInvScale == InvScale::kNinv ? lc.sc_ninv : lc.sc_nqtil;
  u64 v[C::E];
  fold_inv_rounds<Q::LOGM, Q::LOGE, LOGN, Mode, false>(ctx, P, pre, lc, poly, limb, v, sm, tw, tau, f, 2 * q, sc, root,
                                                       rank * Q::M);
  __syncthreads();   // the last round's reads are done
#pragma unroll
  for (int l = 0; l < C::E; ++l) sm[ph(tau + l * C::T)] = fold_s(v[l], f);
  const uint4 w2 = __ldg(tw + 2), w3 = __ldg(tw + 3), k = sc[0], wk = sc[1];
  const u64* y[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) y[i] = cl.map_shared_rank(sm, i);
  cl.sync();
#pragma unroll
  for (int l = 0; l < C::E / 4; ++l) {
    const int p = rank * (Q::M / 4) + tau + l * C::T, at = ph(p);
    const u64 y0 = y[0][at], y1 = y[1][at], y2 = y[2][at], y3 = y[3][at];
    const u64 a0 = y0 + y1, a1 = mul_split(0, y0 - y1, w2, f);
    const u64 a2 = y2 + y3, a3 = mul_split(0, y2 - y3, w3, f);
    const u64 x[4] = {mul_split(2 * q, a0 + a2, k, f), mul_split(2 * q, a1 + a3, k, f),
                      mul_split(2 * q, a0 - a2, wk, f), mul_split(2 * q, a1 - a3, wk, f)};
#pragma unroll
    for (int i = 0; i < 4; ++i)
      Mode::template store<1 << LOGN>(ctx, P, lc, poly, limb, p + i * Q::M, csub(fold_u(x[i], f), q));
  }
  cl.sync();   // the other CTAs have finished reading this one's shared memory
}

// Launch shape of either engine.
template <int LOGN, int LOGE, bool FOLD>
struct KCfg {
  static constexpr int T = (1 << LOGN) >> LOGE;
  static constexpr size_t SMEM = FOLD ? FCfg<LOGN, LOGE>::SMEM : NttCfg<LOGN, LOGE>::SMEM;
  static constexpr int MIN_BLOCKS = FOLD ? FCfg<LOGN, LOGE>::MIN_BLOCKS : NttCfg<LOGN, LOGE>::MIN_BLOCKS;
};

template <int LOGN, int LOGE, class Mode, bool FOLD>
__device__ __forceinline__ void fwd_any(const DevCtx& ctx, const typename Mode::Params& P, int poly, int limb,
                                        u64* sm) {
  if constexpr (FOLD)
    ntt_fwd_run_fold<LOGN, LOGE, Mode>(ctx, P, poly, limb, sm);
  else
    ntt_fwd_run<LOGN, LOGE, Mode>(ctx, P, poly, limb, sm);
}

template <int LOGN, int LOGE, class Mode, bool FOLD>
__device__ __forceinline__ void inv_any(const DevCtx& ctx, const typename Mode::Params& P, int poly, int limb,
                                        u64* sm) {
  if constexpr (FOLD)
    ntt_inv_run_fold<LOGN, LOGE, Mode>(ctx, P, poly, limb, sm);
  else
    ntt_inv_run<LOGN, LOGE, Mode>(ctx, P, poly, limb, sm);
}

// Modes whose input is one contiguous polynomial per (poly, limb): each CTA asks
// L2 for the input of the CTA P.ahead launch positions later (about a wave on),
// so that CTA's first loads hit L2.
template <class M, class = void>
struct PrefetchAhead : std::false_type {};
template <class M>
struct PrefetchAhead<M, std::void_t<decltype(M::kPrefetchAhead)>> : std::bool_constant<M::kPrefetchAhead> {};

template <int N, class Mode>
__device__ __forceinline__ void prefetch_ahead(const DevCtx& ctx, const typename Mode::Params& P, int first) {
  if constexpr (PrefetchAhead<Mode>::value) {
    if (threadIdx.x == 0 && P.ahead > 0) {
      const long long next = (long long)blockIdx.x + (long long)blockIdx.y * gridDim.x + P.ahead;
      const long long y = next / gridDim.x;
      if (y < (long long)gridDim.y) Mode::template prefetch<N>(ctx, P, first + (int)(next % gridDim.x), (int)y);
    }
  }
}

// CTA (x, limb) transforms polynomial first + x; MB CTAs per SM.
template <int LOGN, int LOGE, class Mode, bool FOLD, int MB = KCfg<LOGN, LOGE, FOLD>::MIN_BLOCKS>
__global__ void __launch_bounds__(KCfg<LOGN, LOGE, FOLD>::T, MB)
    k_ntt_fwd(DevCtx ctx, typename Mode::Params P, int first) {
  extern __shared__ __align__(16) u64 sm[];
  prefetch_ahead<1 << LOGN, Mode>(ctx, P, first);
  fwd_any<LOGN, LOGE, Mode, FOLD>(ctx, P, first + (int)blockIdx.x, blockIdx.y, sm);
}

template <int LOGN, int LOGE, class Mode, bool FOLD, int MB = KCfg<LOGN, LOGE, FOLD>::MIN_BLOCKS>
__global__ void __launch_bounds__(KCfg<LOGN, LOGE, FOLD>::T, MB)
    k_ntt_inv(DevCtx ctx, typename Mode::Params P, int first) {
  extern __shared__ __align__(16) u64 sm[];
  prefetch_ahead<1 << LOGN, Mode>(ctx, P, first);
  inv_any<LOGN, LOGE, Mode, FOLD>(ctx, P, first + (int)blockIdx.x, blockIdx.y, sm);
}

// Cluster (x / 4, limb) of four CTAs transforms polynomial first + x / 4.
template <int LOGN, class Mode, bool INV>
__global__ void __launch_bounds__((1 << LOGN) / 32) k_ntt_quad(const __grid_constant__ DevCtx ctx,
                                                               const __grid_constant__ typename Mode::Params P,
                                                               int first) {
  extern __shared__ __align__(16) u64 sm[];
  if constexpr (INV)
    quad_inv<LOGN, Mode>(ctx, P, first + (int)(blockIdx.x >> 2), blockIdx.y, sm);
  else
    quad_fwd<LOGN, Mode>(ctx, P, first + (int)(blockIdx.x >> 2), blockIdx.y, sm);
}

// Multi-plan variants: CTA (blockIdx.x, limb) transforms polynomial items[x].y
// of the plan items[x].x with that plan's parameters; `step` (device word,
// nullable) re-keys the randomness of each replay (Mode::rebase).
template <int LOGN, int LOGE, class Mode, bool FOLD>
__global__ void __launch_bounds__(KCfg<LOGN, LOGE, FOLD>::T, KCfg<LOGN, LOGE, FOLD>::MIN_BLOCKS)
    k_ntt_fwd_multi(DevCtx ctx, const typename Mode::Params* __restrict__ Ps, const int2* __restrict__ items,
                    const u64* step) {
  extern __shared__ __align__(16) u64 sm[];
  const int2 it = items[blockIdx.x];
  typename Mode::Params P = Ps[it.x];
  Mode::rebase(P, step ? *step : 0ull);
  fwd_any<LOGN, LOGE, Mode, FOLD>(ctx, P, it.y, blockIdx.y, sm);
}

template <int LOGN, int LOGE, class Mode, bool FOLD>
__global__ void __launch_bounds__(KCfg<LOGN, LOGE, FOLD>::T, KCfg<LOGN, LOGE, FOLD>::MIN_BLOCKS)
    k_ntt_inv_multi(DevCtx ctx, const typename Mode::Params* __restrict__ Ps, const int2* __restrict__ items,
                    const u64* step) {
  extern __shared__ __align__(16) u64 sm[];
  const int2 it = items[blockIdx.x];
  typename Mode::Params P = Ps[it.x];
  Mode::rebase(P, step ? *step : 0ull);
  inv_any<LOGN, LOGE, Mode, FOLD>(ctx, P, it.y, blockIdx.y, sm);
}

// ------------------------------------------------------------------ fused modes
__device__ __forceinline__ size_t limb_off(int poly, int limb, int L, int n) {
  return ((size_t)poly * L + limb) * n;
}
__device__ __forceinline__ size_t ct_off(int poly, int comp, int limb, int L, int n) {
  return (((size_t)poly * 2 + comp) * L + limb) * n;
}

// What a mode keeps per polynomial for its prologue (Mode::Pre).
struct NoPre {
  template <class P>
  __device__ __forceinline__ NoPre(const DevCtx&, const P&, int) {}
};
struct WindowPre {
  Window win;
  template <class P>
  __device__ __forceinline__ WindowPre(const DevCtx&, const P& p, int poly) : win(p.pk, p.ac, poly, p.ac.ptr) {}
};

// The split engine (SPLIT) takes prologue values as signed lazy residues in about
// [-1/2, 1] (units of 2^b), the Shoup engine canonical ones.

// In-place transform of [count][L][N] polynomials.
struct ModeRaw {
  static constexpr InvScale kInvScale = InvScale::kNinv;
  static constexpr bool kHeavyLoad = false;
  static constexpr bool kQuad = false;
  static constexpr int kLoadUnroll = 32;
  static constexpr int kEpilogueUnroll = 16;
  static constexpr bool kPrefetchAhead = true;
  struct Params {
    u64* polys;
    int ahead = 0;   // CTAs ahead whose input each CTA asks L2 to fetch (0: none)
  };
  using Pre = NoPre;
  static __device__ __forceinline__ void rebase(Params&, u64) {}
  // two consecutive slots of an inverse transform (split engine)
  template <int N>
  static __device__ __forceinline__ void load2(const DevCtx& c, const Params& P, const LimbConst&, int poly, int limb,
                                               int e, u64& x0, u64& x1) {
    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(P.polys + limb_off(poly, limb, c.L, N) + e);
    x0 = x.x;
    x1 = x.y;
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx& c, const Params& P, const Pre& pre, const LimbConst&, int poly, int limb,
                                             int e) {
    return P.polys[limb_off(poly, limb, c.L, N) + e];
  }
  template <int N>
  static __device__ __forceinline__ void prefetch(const DevCtx& c, const Params& P, int poly, int limb) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(P.polys + limb_off(poly, limb, c.L, N)),
                 "r"((u32)(N * sizeof(u64)))
                 : "memory");
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ void store2(const DevCtx& c, const Params& P, const LimbConst&, int poly,
                                                int limb, int e, u64 x0, u64 x1) {
    *reinterpret_cast<ulonglong2*>(P.polys + limb_off(poly, limb, c.L, N) + e) = make_ulonglong2(x0, x1);
  }
  template <int N>
  static __device__ __forceinline__ void store(const DevCtx& c, const Params& P, const LimbConst& lc, int poly,
                                               int limb, int e, u64 x) {
    P.polys[limb_off(poly, limb, c.L, N) + e] = x;   // x = N^{-1} INTT, canonical
  }
};

// DO encryption: prologue round(q m / t) + e (m gathered by the packing), epilogue
// c0 = slot - a*s_hat, c1 = a with a sampled in the NTT domain, four coefficients
// per Philox block (one 64-bit word each, uniform_word).
struct ModeEncrypt {
  static constexpr bool kHeavyLoad = true;
  static constexpr bool kQuad = true;
  static constexpr int kLoadUnroll = 8;
  static constexpr int kEpilogueUnroll = 1;   // Philox + four products per quad
  struct Params {
    Packing pk;
    Accessor ac;
    const int8_t* err;        // [count][N]
    const ulonglong2* sk;     // [L][N] (s_hat, companion), [L][N] split s_hat
    u64* ct;                  // [count][2][L][N]
    u64 seed;
  };
  // seed of replay `step` (batched graphs): seed + step * 2^32
  using Pre = WindowPre;
  static __device__ __forceinline__ void rebase(Params& P, u64 step) { P.seed += step << 32; }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx& c, const Params& P, const Pre& pre, const LimbConst& lc, int poly, int,
                                             int e) {
    const u64 m = pre.win.get(P.pk, e) & c.t_mask;
    const int ee = P.err[(size_t)poly * N + e];
    if constexpr (SPLIT) {
      const FoldC f(lc);
      return fold_s(mul_split(scale_extra(m, c) + (i64)ee, m, lc.delta_sp, f), f);
    }
    const u64 r = scale_msg(m, lc, c);
    return ee >= 0 ? add_mod(r, (u64)ee, lc.q) : sub_mod(r, (u64)(-ee), lc.q);
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ void store4(const DevCtx& c, const Params& P, const LimbConst& lc, int poly,
                                                int limb, int e, const u64* x) {
    const Philox4 w = philox4x64((u64)(e >> 2), (u64)poly, (u64)limb, 0ull, P.seed, PENCIL_DOM_A);
    u64 a[4], c0[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const u64 word = uniform_word(w.v[i], e + i, poly, limb, P.seed, PENCIL_DOM_A, lc);
      if constexpr (SPLIT) {
        const FoldC f(lc);
        a[i] = csub(fold_u(word, f), lc.q);
        const uint4 s = __ldg(reinterpret_cast<const uint4*>(P.sk) + (size_t)(c.L + limb) * N + e + i);
        c0[i] = csub(fold_u(x[i] + 2 * lc.q - mul_split(0, a[i], s, f), f), lc.q);
      } else {
        a[i] = reduce64(word, lc);
        const ulonglong2 s = __ldg(P.sk + (size_t)limb * N + e + i);
        c0[i] = sub_mod(x[i], mul_shoup(a[i], s.x, s.y, lc.q), lc.q);
      }
    }
    ulonglong2* d0 = reinterpret_cast<ulonglong2*>(P.ct + ct_off(poly, 0, limb, c.L, N) + e);
    ulonglong2* d1 = reinterpret_cast<ulonglong2*>(P.ct + ct_off(poly, 1, limb, c.L, N) + e);
    d0[0] = make_ulonglong2(c0[0], c0[1]);
    d0[1] = make_ulonglong2(c0[2], c0[3]);
    d1[0] = make_ulonglong2(a[0], a[1]);
    d1[1] = make_ulonglong2(a[2], a[3]);
  }
};

// MO plaintext encoding: centred lift of Z_t values, NTT (short supports,
// e.g. one small kernel block per plaintext, skip the copy-only stages).
struct ModeEncode {
  static constexpr bool kHeavyLoad = true;
  static constexpr bool kQuad = false;
  static constexpr bool kSparse = true;
  static constexpr int kLoadUnroll = 16;
  static constexpr int kEpilogueUnroll = 4;
  struct Params {
    Packing pk;
    Accessor ac;
    u64* pt;   // [count][L][N]
  };
  static __device__ __forceinline__ int support(const Params& P) { return P.pk.support; }
  using Pre = WindowPre;
  static __device__ __forceinline__ void rebase(Params&, u64) {}
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx& c, const Params& P, const Pre& pre, const LimbConst& lc, int poly, int,
                                             int e) {
    const u64 v = pre.win.get(P.pk, e) & c.t_mask;
    const u64 half = (c.t_mask >> 1) + 1;
    if constexpr (SPLIT) return v >= half ? v - (c.t_mask + 1) : v;
    return v >= half ? lc.q - ((c.t_mask + 1) - v) : v;
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ void store2(const DevCtx& c, const Params& P, const LimbConst&, int poly,
                                                int limb, int e, u64 x0, u64 x1) {
    *reinterpret_cast<ulonglong2*>(P.pt + limb_off(poly, limb, c.L, N) + e) = make_ulonglong2(x0, x1);
  }
};

// MO's ciphertext-independent terms of Alg. 1 steps 2-3, one launch for both:
// polynomials [0, n_in) -> out_in = NTT(round(q pi_v(x0) / t)) (added to c0 by the
// multiply-accumulate), [n_in, count) -> out_mask = NTT(round(q s / t)) of the mask
// polynomials (subtracted by the multiply-accumulate's store).
struct ModeMoPrep {
  static constexpr bool kHeavyLoad = true;
  static constexpr bool kQuad = false;
  static constexpr int kLoadUnroll = 16;
  static constexpr int kEpilogueUnroll = 8;
  struct Params {
    Packing pk;
    Accessor ac;
    const u64* mpoly;   // [count - n_in][N] Z_t mask coefficients
    int n_in;
    u64* out_in;        // [n_in][L][N]
    u64* out_mask;      // [count - n_in][L][N]
    u64 seed;           // mask seed (key of the flooding stream)
  };
  // input polynomials' window (the mask polynomials have none)
  struct Pre {
    const char* base = nullptr;
    u32 tl = 0, th = 0, lh = 0;
    __device__ __forceinline__ Pre(const DevCtx&, const Params& P, int poly) {
      if (poly >= P.n_in) return;
      const Window w(P.pk, P.ac, poly, P.ac.ptr);
      base = w.base;
      tl = w.tl;
      th = w.th;
      lh = w.lh;
    }
  };
  static __device__ __forceinline__ void rebase(Params& P, u64 step) { P.seed += step << 32; }   // as the mask's
  // The mask polynomials are contiguous: their words go straight to registers, all of a
  // thread's in flight (1920 beside 90 inputs, N = 8192, three limbs: 504 -> 424 us), and
  // flooding draws one Philox block per four words instead of one per word (a 64 x 2048
  // by 2048 x 1001 layer with flooding: the whole call 1532 -> 1437 us).
  static constexpr bool kDirect = true;
  template <int N>
  static __device__ __forceinline__ const u64* direct(const Params& P, int poly) {
    return poly >= P.n_in ? P.mpoly + (size_t)(poly - P.n_in) * N : nullptr;
  }
  static __device__ __forceinline__ bool noisy(const DevCtx& c) { return c.flood_bits != 0; }
  // flooding noise f (uniform in [-2^b, 2^b)) of returned ciphertext poly - n_in at words
  // e .. e + 3, and what it adds: Delta s - f
  static __device__ __forceinline__ Philox4 noise(const Params& P, int poly, int e) {
    return philox4x64((u64)(e >> 2), (u64)(poly - P.n_in), 0ull, 0ull, P.seed, PENCIL_DOM_FLOOD);
  }
  static __device__ __forceinline__ i64 noise_add(const DevCtx& c, u64 w) {
    return (i64)((1ull << c.flood_bits) - (w & ((2ull << c.flood_bits) - 1)));
  }
  // (|add| <= 2^62: inside the signed range with the product)
  static __device__ __forceinline__ u64 direct_value(const DevCtx& c, u64 m, i64 add, const LimbConst& lc,
                                                     const FoldC& f) {
    return fold_s(mul_split(scale_extra(m, c) + add, m, lc.delta_sp, f), f);
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx& c, const Params& P, const Pre& pre, const LimbConst& lc,
                                             int poly, int, int e) {
    i64 add = 0;
    u64 m;
    if (poly < P.n_in) {
      m = Window(pre.base, pre.tl, pre.th, pre.lh).get(P.pk, e) & c.t_mask;
    } else {
      m = P.mpoly[(size_t)(poly - P.n_in) * N + e];
      if (c.flood_bits) add = noise_add(c, philox_word(noise(P, poly, e), e & 3));
    }
    if constexpr (SPLIT) {
      const FoldC f(lc);
      return direct_value(c, m, add, lc, f);
    }
    const u64 r = scale_msg(m, lc, c);
    if (!c.flood_bits) return r;   // (uniform: the reductions below were 3 % of the whole call)
    return add >= 0 ? add_mod(r, reduce64((u64)add, lc), lc.q) : sub_mod(r, reduce64((u64)-add, lc), lc.q);
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ void store2(const DevCtx& c, const Params& P, const LimbConst&, int poly,
                                                int limb, int e, u64 x0, u64 x1) {
    u64* dst = poly < P.n_in ? P.out_in + limb_off(poly, limb, c.L, N)
                             : P.out_mask + limb_off(poly - P.n_in, limb, c.L, N);
    *reinterpret_cast<ulonglong2*>(dst + e) = make_ulonglong2(x0, x1);
  }
};

__device__ __forceinline__ u64 shoup_companion(u64 w, u64 q) {
  return (u64)((((unsigned __int128)w) << 64) / q);
}

// Word `at` of a key of `rows` x n values: with its Shoup companion and, in contexts that
// have the split butterflies, as a split twiddle behind all of those (mul_split).
__device__ __forceinline__ void put_key(const DevCtx& c, ulonglong2* key, int rows, size_t at, int n, u64 x,
                                        const LimbConst& lc) {
  key[at] = make_ulonglong2(x, shoup_companion(x, lc.q));
  if (!c.tw_fwd_f) return;
  const u64 half = lc.q >> 1, y = reduce128(x >> 32, x << 32, lc);
  const i64 a = x > half ? (i64)(x - lc.q) : (i64)x, b = y > half ? (i64)(y - lc.q) : (i64)y;
  const u64 m = (1ull << lc.sb) - 1ull;
  reinterpret_cast<uint4*>(key)[(size_t)rows * n + at] =
      make_uint4((u32)((u64)a & m), (u32)(a >> lc.sb), (u32)((u64)b & m), (u32)(b >> lc.sb));
}

// DO key generation: ternary s, NTT, stored for both product forms.
struct ModeKeygen {
  static constexpr bool kHeavyLoad = true;
  static constexpr bool kQuad = false;
  static constexpr int kLoadUnroll = 4;
  static constexpr int kEpilogueUnroll = 1;
  struct Params {
    u64 seed;
    ulonglong2* sk;   // [L][N] with companions, then [L][N] split
  };
  using Pre = NoPre;
  static __device__ __forceinline__ void rebase(Params&, u64) {}
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx&, const Params& P, const Pre& pre, const LimbConst& lc, int, int, int e) {
    const Philox4 w = philox4x64((u64)(e >> 2), 0ull, 0ull, 0ull, P.seed, PENCIL_DOM_SECRET);
    const u64 r = w.v[e & 3] % 3ull;
    return r == 0 ? lc.q - 1 : r - 1;
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ void store2(const DevCtx& c, const Params& P, const LimbConst& lc, int, int limb,
                                                int e, u64 x0, u64 x1) {
    put_key(c, P.sk, c.L, limb * N + e, N, x0, lc);
    put_key(c, P.sk, c.L, limb * N + e + 1, N, x1, lc);
  }
};

__device__ __forceinline__ u64 lift_small(int v, u64 q) { return v >= 0 ? (u64)v : q - (u64)(-v); }
__device__ __forceinline__ u64 neg_mod(u64 v, u64 q) { return v ? q - v : 0; }

// DO public key (BFV as in Fan-Vercauteren): x = NTT(e) of the sampled error;
// p1 = a, uniform in the NTT domain from Philox (key (seed, 7), counter
// (i/4, 0, limb, 0), word i%4; uniform_word); p0 = -(a s) - x.  Both stored as
// put_key stores them: key[comp][L][N].
struct ModePkKeygen {
  static constexpr bool kHeavyLoad = true;
  static constexpr bool kQuad = true;
  static constexpr int kLoadUnroll = 8;
  static constexpr int kEpilogueUnroll = 1;
  struct Params {
    const int8_t* err;       // [N]
    const ulonglong2* sk;    // [L][N]
    ulonglong2* key;         // [2][L][N] with companions, then [2][L][N] split
    u64 seed;
  };
  using Pre = NoPre;
  static __device__ __forceinline__ void rebase(Params&, u64) {}
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx&, const Params& P, const Pre& pre, const LimbConst& lc, int, int, int e) {
    return lift_small(P.err[e], lc.q);
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ void store4(const DevCtx& c, const Params& P, const LimbConst& lc, int, int limb,
                                                int e, const u64* x) {
    const Philox4 w = philox4x64((u64)(e >> 2), 0ull, (u64)limb, 0ull, P.seed, PENCIL_DOM_PK_A);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const u64 a = reduce64(uniform_word(w.v[i], e + i, 0, limb, P.seed, PENCIL_DOM_PK_A, lc), lc);
      const ulonglong2 s = __ldg(P.sk + (size_t)limb * N + e + i);
      const u64 p0 = neg_mod(add_mod(mul_shoup(a, s.x, s.y, lc.q), x[i], lc.q), lc.q);
      put_key(c, P.key, 2 * c.L, (size_t)limb * N + e + i, N, p0, lc);
      put_key(c, P.key, 2 * c.L, (size_t)(c.L + limb) * N + e + i, N, a, lc);
    }
  }
};

// Public-key encryption, first pass: NTT(u) of each ciphertext's ternary u.
struct ModePkU {
  static constexpr bool kHeavyLoad = false;
  static constexpr bool kQuad = false;
  static constexpr int kLoadUnroll = 16;
  static constexpr int kEpilogueUnroll = 8;
  struct Params {
    const int8_t* u;   // [ct][N]
    u64* u_hat;        // [ct][L][N]
  };
  using Pre = NoPre;
  static __device__ __forceinline__ void rebase(Params&, u64) {}
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx&, const Params& P, const Pre& pre, const LimbConst& lc, int poly, int,
                                             int e) {
    const int v = P.u[(size_t)poly * N + e];
    if constexpr (SPLIT) return (u64)(i64)v;
    return lift_small(v, lc.q);
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ void store2(const DevCtx& c, const Params& P, const LimbConst&, int poly,
                                                int limb, int e, u64 x0, u64 x1) {
    *reinterpret_cast<ulonglong2*>(P.u_hat + limb_off(poly, limb, c.L, N) + e) = make_ulonglong2(x0, x1);
  }
};

// Public-key encryption, second pass, over polynomials 2 ct + comp:
//   comp 0: NTT(Delta m + e1) + NTT(u) p0,   comp 1: NTT(e2) + NTT(u) p1,
// written straight into ciphertext ct (whose [2][L][N] layout makes
// polynomial 2 ct + comp the component's slot).
struct ModeEncryptPk {
  static constexpr bool kHeavyLoad = true;
  static constexpr bool kQuad = false;
  static constexpr int kLoadUnroll = 8;
  static constexpr int kEpilogueUnroll = 4;
  struct Params {
    Packing pk;
    Accessor ac;
    const int8_t* e1;          // [ct][N]
    const int8_t* e2;          // [ct][N]
    const u64* u_hat;          // [ct][L][N]
    const ulonglong2* key;     // [2][L][N] with companions, then [2][L][N] split
    u64* ct;                   // [ct][2][L][N]
  };
  struct Pre {
    Window win;
    __device__ __forceinline__ Pre(const DevCtx&, const Params& P, int poly) : win(P.pk, P.ac, poly >> 1, P.ac.ptr) {}
  };
  static __device__ __forceinline__ void rebase(Params&, u64) {}
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx& c, const Params& P, const Pre& pre, const LimbConst& lc, int poly, int,
                                             int e) {
    const int ct = poly >> 1;
    if (poly & 1) {
      const int e2 = P.e2[(size_t)ct * N + e];
      if constexpr (SPLIT) return (u64)(i64)e2;
      return lift_small(e2, lc.q);
    }
    const u64 m = pre.win.get(P.pk, e) & c.t_mask;
    const int ee = P.e1[(size_t)ct * N + e];
    if constexpr (SPLIT) {
      const FoldC f(lc);
      return fold_s(mul_split(scale_extra(m, c) + (i64)ee, m, lc.delta_sp, f), f);
    }
    const u64 r = scale_msg(m, lc, c);
    return ee >= 0 ? add_mod(r, (u64)ee, lc.q) : sub_mod(r, (u64)(-ee), lc.q);
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ void store2(const DevCtx& c, const Params& P, const LimbConst& lc, int poly,
                                                int limb, int e, u64 x0, u64 x1) {
    const int ct = poly >> 1, comp = poly & 1;
    const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(P.u_hat + limb_off(ct, limb, c.L, N) + e);
    const size_t at = (size_t)(comp * c.L + limb) * N + e;
    u64 y0, y1;
    if constexpr (SPLIT) {
      const FoldC f(lc);
      const uint4* key = reinterpret_cast<const uint4*>(P.key) + 2 * (size_t)c.L * N + at;
      y0 = csub(fold_u(mul_split(x0 + lc.q, u.x, __ldg(key), f), f), lc.q);
      y1 = csub(fold_u(mul_split(x1 + lc.q, u.y, __ldg(key + 1), f), f), lc.q);
    } else {
      const ulonglong2 k0 = __ldg(P.key + at), k1 = __ldg(P.key + at + 1);
      y0 = add_mod(x0, mul_shoup(u.x, k0.x, k0.y, lc.q), lc.q);
      y1 = add_mod(x1, mul_shoup(u.y, k1.x, k1.y, lc.q), lc.q);
    }
    *reinterpret_cast<ulonglong2*>(P.ct + ct_off(ct, comp, limb, c.L, N) + e) = make_ulonglong2(y0, y1);
  }
};

// DO decryption, first half: x = INTT(c0 + c1 * s_hat); stores y = x * qtilde mod q_j
// (the INTT's N^{-1} and qtilde are one constant).
// With skip_c0 (decryption of the compact send form) only c1 * s is transformed;
// the output coefficients' c0 is added by the combine kernel.
struct ModeDecrypt {
  static constexpr InvScale kInvScale = InvScale::kNqtil;
  static constexpr bool kHeavyLoad = true;
  static constexpr bool kQuad = false;
  static constexpr int kLoadUnroll = 8;
  static constexpr int kEpilogueUnroll = 16;
  struct Params {
    const u64* ct;          // [count][2][L][N]
    const ulonglong2* sk;   // [L][N] with companions, then [L][N] split
    u64* out;               // [count][L][N]
    int skip_c0;
    const unsigned char* groups;   // ModeDecryptFew: the output packing's (Packing::groups)
  };
  using Pre = NoPre;
  static __device__ __forceinline__ void rebase(Params&, u64) {}
  template <int N>
  static __device__ __forceinline__ void load2(const DevCtx& c, const Params& P, const LimbConst& lc, int poly,
                                               int limb, int e, u64& x0, u64& x1) {
    const FoldC f(lc);
    const ulonglong2 c1 = __ldg(reinterpret_cast<const ulonglong2*>(P.ct + ct_off(poly, 1, limb, c.L, N) + e));
    const uint4* key = reinterpret_cast<const uint4*>(P.sk) + (size_t)(c.L + limb) * N + e;
    const uint4 s0 = __ldg(key), s1 = __ldg(key + 1);
    if (P.skip_c0) {
      x0 = mul_split(0, c1.x, s0, f);
      x1 = mul_split(0, c1.y, s1, f);
    } else {
      const ulonglong2 c0 = __ldg(reinterpret_cast<const ulonglong2*>(P.ct + ct_off(poly, 0, limb, c.L, N) + e));
      x0 = fold_s(mul_split(c0.x, c1.x, s0, f), f);
      x1 = fold_s(mul_split(c0.y, c1.y, s1, f), f);
    }
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx& c, const Params& P, const Pre& pre, const LimbConst& lc, int poly,
                                             int limb, int e) {
    const u64 c1 = __ldg(P.ct + ct_off(poly, 1, limb, c.L, N) + e);
    if constexpr (SPLIT) {   // c0 + c1 s in [-0.6, 2.6], folded
      const FoldC f(lc);
      const uint4 s = __ldg(reinterpret_cast<const uint4*>(P.sk) + (size_t)(c.L + limb) * N + e);
      // one product for both forms: a branch around a second one kept the loads of different
      // words apart (256 polynomials at N = 8192 with radix 2^5: 125 us, 89 like this)
      const u64 c0 = P.skip_c0 ? 0 : __ldg(P.ct + ct_off(poly, 0, limb, c.L, N) + e);
      return fold_s(mul_split(c0, c1, s, f), f);
    }
    const ulonglong2 s = __ldg(P.sk + (size_t)limb * N + e);
    const u64 c1s = mul_shoup(c1, s.x, s.y, lc.q);
    if (P.skip_c0) return c1s;
    return add_mod(__ldg(P.ct + ct_off(poly, 0, limb, c.L, N) + e), c1s, lc.q);
  }
  template <int N>
  static __device__ __forceinline__ void store(const DevCtx& c, const Params& P, const LimbConst& lc, int poly,
                                               int limb, int e, u64 x) {
    P.out[limb_off(poly, limb, c.L, N) + e] = x;   // x = N^{-1} qtil INTT, canonical
  }
};

// The same for polynomials of which many groups of 32 coefficients carry no output
// (compact_skips): the CRT pass reads no residue of those, and none is written.
struct ModeDecryptFew : ModeDecrypt {
  static constexpr bool kFewOutputs = true;
  static __device__ __forceinline__ bool occupied(const Params& P, int group) { return __ldg(P.groups + group) != 0; }
};

// MO, compact send form of returned ciphertexts: INTT(c0) and, at the
// coefficients carrying output element flat, c0c[limb][flat] = that coefficient
// (the rest is dropped).
struct ModeCompact {
  static constexpr InvScale kInvScale = InvScale::kNinv;
  static constexpr bool kHeavyLoad = false;
  static constexpr bool kQuad = false;
  static constexpr int kLoadUnroll = 16;
  static constexpr int kEpilogueUnroll = 16;
  struct Params {
    const u64* ct;          // [count][2][L][N]
    Packing pk;             // output packing
    Accessor ac;            // output layout
    u64* c0c;               // [L][out_elems]
    long long out_elems;
  };
  using Pre = NoPre;
  static __device__ __forceinline__ void rebase(Params&, u64) {}
  template <int N>
  static __device__ __forceinline__ void load2(const DevCtx& c, const Params& P, const LimbConst&, int poly, int limb,
                                               int e, u64& x0, u64& x1) {
    const ulonglong2 x = __ldg(reinterpret_cast<const ulonglong2*>(P.ct + ct_off(poly, 0, limb, c.L, N) + e));
    x0 = x.x;
    x1 = x.y;
  }
  template <int N, bool SPLIT>
  static __device__ __forceinline__ u64 load(const DevCtx& c, const Params& P, const Pre& pre, const LimbConst&, int poly, int limb,
                                             int e) {
    return __ldg(P.ct + ct_off(poly, 0, limb, c.L, N) + e);
  }
  template <int N>
  static __device__ __forceinline__ void store(const DevCtx&, const Params& P, const LimbConst& lc, int poly,
                                               int limb, int e, u64 x) {
    const i64 flat = Window(P.pk, P.ac, poly, nullptr).index(P.pk, e);
    if (flat >= 0) P.c0c[(size_t)limb * P.out_elems + flat] = x;   // x = N^{-1} INTT, canonical
  }
};

// The same for polynomials of which many groups of 32 coefficients carry no output
// (compact_skips).
struct ModeCompactFew : ModeCompact {
  static constexpr bool kFewOutputs = true;
  static __device__ __forceinline__ bool occupied(const Params& P, int group) { return __ldg(P.pk.groups + group) != 0; }
};

// Whether a launch of `count` polynomials runs on clusters of four CTAs: forward while
// every CTA has an SM of its own (its first two stages cost three products a word instead
// of one), inverse, which does no more work, up to two per SM.  Measured (us, clusters /
// one CTA each; N = 8192): forward 8 transforms 9.8 / 12.2, 38 12.1 / 12.1, 76 15.3 /
// 12.2; inverse 8 7.4 / 12.8, 76 11.6 / 12.9, 120 14.3 / 12.9.  N = 16384: forward 8 12.9
// / 21.8, 38 19.9 / 22.0, 76 27.5 / 22.4; inverse 76 22.4 / 24.1, 152 35.4 / 24.5.
// N = 4096 (L = 2): inverse 3 transforms 5.5 / 7.2; encryption 10.3 / 13.6, encoding 6.7 / 7.3,
// preparation 13.9 / 15.5; the bare forward transform, whose prologue and epilogue leave the
// CTAs nothing else to share, 7.5 / 6.3: it alone stays in one CTA.
inline bool quad_wins(const DevCtx& ctx, long long count, bool inverse) {
  return ctx.ntt_arith && ctx.ntt_loge == 4 && 4 * count * ctx.L <= (inverse ? 2 : 1) * ctx.sms;
}

// Whether a launch of 256-thread transforms (N = 4096, radix 2^4) runs four to an SM with 64
// registers a thread (some spill a word or two) instead of two with up to 120: once there are
// enough of them, issue is what bounds it and 32 warps hide more than 16; a launch that fits
// the SMs in one go is each transform's latency, which the registers shorten.  Measured (us, two /
// four per SM): raw forward 2.6 transforms per SM 26.1 / 26.2, 3.9 30.7 / 30.3, 5.1 39.1 /
// 38.2, 13.8 75.1 / 68.2, 59 279 / 247; raw inverse 3.9 33.9 / 34.9, 5.1 43.2 / 42.8, 7.9
// 52.5 / 52.9, 59 310 / 289; encoding 3.4 27.8 / 26.4, 13.5 63.5 / 55.1; MO preparation 18.5
// 180 / 154; decryption 4.6 65.7 / 58.5, 9.3 122 / 101.
inline bool many_small(const DevCtx& ctx, long long count, bool inverse) {
  return count * ctx.L > (inverse ? 4ll : 3ll) * ctx.sms;
}

// Whether a launch of 512-thread transforms (N = 8192, radix 2^4) that gives no SM two of them
// is compiled for one CTA per SM, with up to 128 registers a thread instead of 64: there is
// no second CTA whose warps hide a transform's latency (us, two per SM / one: raw forward 75
// transforms 11.7 / 10.9, 120 11.8 / 10.9; raw inverse 120 12.4 / 12.0; encryption 96 23.5 /
// 22.7; decryption 120 18.7 / 18.1; compact form 120 14.6 / 13.5; 240 transforms, two on an
// SM, forward 19.9 / 20.6).
inline bool lone(const DevCtx& ctx, long long count) { return count * ctx.L <= ctx.sms; }

// Host-side launcher; explicitly instantiated per LOGN and engine in ntt12.cu /
// ntt13.cu / ntt14.cu (Shoup) and ntt12f.cu / ntt13f.cu / ntt14f.cu (split products).
template <int LOGN, int LOGE, class Mode, bool INV, bool FOLD>
cudaError_t launch_ntt(const DevCtx& ctx, const typename Mode::Params& P, int first, int count, cudaStream_t s) {
  using C = KCfg<LOGN, LOGE, FOLD>;
  if (count <= 0) return cudaSuccess;
  const dim3 grid((unsigned)count, (unsigned)ctx.L);
  if constexpr (FOLD && LOGE == 4) {
    if (quad_wins(ctx, count, INV) && !(LOGN == 12 && std::is_same_v<Mode, ModeRaw> && !INV)) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(4 * (unsigned)count, (unsigned)ctx.L);
      cfg.blockDim = dim3((1 << LOGN) / 32);
      cfg.dynamicSmemBytes = Quad<LOGN>::C::SMEM;
      cfg.stream = s;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = 4;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      return cudaLaunchKernelEx(&cfg, k_ntt_quad<LOGN, Mode, INV>, ctx, P, first);
    }
  }
  auto launch = [&](auto kernel) {
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (err != cudaSuccess) return err;
    kernel<<<grid, C::T, C::SMEM, s>>>(ctx, P, first);
    return cudaGetLastError();
  };
  if constexpr (FOLD && LOGN == 12 && LOGE == 4) {
    if (many_small(ctx, count, INV)) {
      if constexpr (INV)
        return launch(k_ntt_inv<LOGN, LOGE, Mode, FOLD, 4>);
      else
        return launch(k_ntt_fwd<LOGN, LOGE, Mode, FOLD, 4>);
    }
  }
  if constexpr (FOLD && LOGN == 13 && LOGE == 4) {
    if (lone(ctx, count)) {
      if constexpr (INV)
        return launch(k_ntt_inv<LOGN, LOGE, Mode, FOLD, 1>);
      else
        return launch(k_ntt_fwd<LOGN, LOGE, Mode, FOLD, 1>);
    }
  }
  if constexpr (INV)
    return launch(k_ntt_inv<LOGN, LOGE, Mode, FOLD>);
  else
    return launch(k_ntt_fwd<LOGN, LOGE, Mode, FOLD>);
}

template <int LOGN, int LOGE, class Mode, bool INV, bool FOLD>
cudaError_t launch_ntt_multi(const DevCtx& ctx, const typename Mode::Params* Ps, const int2* items, long long count,
                             const u64* step, cudaStream_t s) {
  using C = KCfg<LOGN, LOGE, FOLD>;
  if (count <= 0) return cudaSuccess;
  if (count > 2147483647ll) return cudaErrorInvalidValue;
  cudaError_t err;
  dim3 grid((unsigned)count, (unsigned)ctx.L);
  if constexpr (INV) {
    err = cudaFuncSetAttribute(k_ntt_inv_multi<LOGN, LOGE, Mode, FOLD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)C::SMEM);
    if (err != cudaSuccess) return err;
    k_ntt_inv_multi<LOGN, LOGE, Mode, FOLD><<<grid, C::T, C::SMEM, s>>>(ctx, Ps, items, step);
  } else {
    err = cudaFuncSetAttribute(k_ntt_fwd_multi<LOGN, LOGE, Mode, FOLD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)C::SMEM);
    if (err != cudaSuccess) return err;
    k_ntt_fwd_multi<LOGN, LOGE, Mode, FOLD><<<grid, C::T, C::SMEM, s>>>(ctx, Ps, items, step);
  }
  return cudaGetLastError();
}

#define PENCIL_NTT_INST1(SPEC, LOGN, LOGE, MODE, INV, FOLD)                                                    \
  SPEC template cudaError_t launch_ntt<LOGN, LOGE, MODE, INV, FOLD>(const DevCtx&, const MODE::Params&, int, int, \
                                                                    cudaStream_t);                             \
  SPEC template cudaError_t launch_ntt_multi<LOGN, LOGE, MODE, INV, FOLD>(const DevCtx&, const MODE::Params*,     \
                                                                          const int2*, long long, const u64*,   \
                                                                          cudaStream_t);
#define PENCIL_NTT_INST_E(SPEC, LOGN, LOGE, FOLD)                \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeRaw, false, FOLD)       \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeRaw, true, FOLD)        \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeEncrypt, false, FOLD)   \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeEncode, false, FOLD)    \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeMoPrep, false, FOLD)    \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeKeygen, false, FOLD)    \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModePkKeygen, false, FOLD)  \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModePkU, false, FOLD)       \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeEncryptPk, false, FOLD) \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeCompact, true, FOLD)    \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeCompactFew, true, FOLD) \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeDecrypt, true, FOLD)    \
  PENCIL_NTT_INST1(SPEC, LOGN, LOGE, ModeDecryptFew, true, FOLD)
// Radix 2^4 and 2^5 register blocks for one N and one engine.
#define PENCIL_NTT_INSTANTIATE(SPEC, LOGN, FOLD) \
  PENCIL_NTT_INST_E(SPEC, LOGN, 4, FOLD)         \
  PENCIL_NTT_INST_E(SPEC, LOGN, 5, FOLD)

}  // namespace pencil
