// Launches of the tensor-core multiply-accumulate (mac_mma.cuh).
#include <algorithm>

#include "mac_mma.cuh"

namespace pencil {

// CTA (output block, slot block); output blocks fastest, so the CTAs running at one
// time read the same operand rows (L2).
template <bool DUAL, int MT, int NT>
__global__ void __launch_bounds__(MMA_THREADS, 4) k_mac_mma(const __grid_constant__ DevCtx ctx,
                                                            const __grid_constant__ MacParams P, int ntiles) {
  extern __shared__ __align__(16) u64 sm[];
  const int mb = blockIdx.x / ntiles;
  mac_mma_block<DUAL, MT, NT>(ctx, P, P.m_base + mb * MT, ((int)blockIdx.x - mb * ntiles) * NT,
                              blockIdx.y * MMA_LANES, sm);
}

template <bool DUAL, int MT, int NT>
static cudaError_t launch(const DevCtx& ctx, const MacParams& P0, cudaStream_t s) {
  using T = MmaTile<DUAL, MT, NT>;
  const int stages = P0.K > T::KC ? 2 : 1;
  const size_t smem = T::bytes(stages);
  // The attribute belongs to the function, not to this launch: every caller sets the same
  // (two-stage) value, so that a thread with one stage cannot lower it between another
  // thread's call here and its launch with two.
  const cudaError_t e =
      cudaFuncSetAttribute(k_mac_mma<DUAL, MT, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::bytes(2));
  if (e != cudaSuccess) return e;
  MacParams P = P0;
  const int ntiles = (P0.NC + NT - 1) / NT;
  const long long step = std::max<long long>(1, 2147483647ll / ntiles) * MT;   // output rows of one launch
  for (long long base = P0.m_base; base < P0.M; base += step) {
    P.m_base = (int)base;
    P.M = (int)std::min<long long>(P0.M, base + step);
    const dim3 grid((unsigned)((P.M - P.m_base + MT - 1) / MT) * (unsigned)ntiles, (unsigned)(P0.lanes / MMA_LANES));
    k_mac_mma<DUAL, MT, NT><<<grid, MMA_THREADS, smem, s>>>(ctx, P, ntiles);
    const cudaError_t e2 = cudaGetLastError();
    if (e2 != cudaSuccess) return e2;
  }
  return cudaSuccess;
}

// Output blocks: 16 rows where there are more than 8 and one chunk holds all input
// blocks (M = 10, K = 16, NC = 16: 96 us against 111 us with 8 rows) and for Alg. 2
// (M = 64, K = 32, NC = 43: 4.08 ms against 4.34 ms); 8 rows where two stages are
// needed (M = 16, K = 32, NC = 32: 399 us against 535 us: 4 CTAs per SM instead of 2).
cudaError_t launch_mac_mma(const DevCtx& ctx, const MacParams& P, bool dual, cudaStream_t s) {
  const int rows = P.M - P.m_base;
  if (dual) return rows > 8 ? launch<true, 16, 16>(ctx, P, s) : launch<true, 8, 16>(ctx, P, s);
  if (rows > 8 && P.K <= 16) return launch<false, 16, 16>(ctx, P, s);
  return launch<false, 8, 16>(ctx, P, s);
}

}  // namespace pencil
