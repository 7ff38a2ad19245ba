// Combination kernels that take the last chunk first, bf16 gradients, K = 1..16,
// fp32 or bf16 output.
#include "combine_impl.cuh"

namespace bkmoo {
BKMOO_COMBINE_TABLE(BKMOO_BF16);
const void* combine_fn_bf16(int K, int dtype_out) { return kCombineTable[K - 1][dtype_out]; }
}  // namespace bkmoo
