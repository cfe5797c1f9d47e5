// Instantiates the fused NTT / INTT kernels for N = 2^14 (signed split-product butterflies, q = 2^b - c).
#include "ntt.cuh"
namespace pencil {
PENCIL_NTT_INSTANTIATE(, 14, true)
}  // namespace pencil
