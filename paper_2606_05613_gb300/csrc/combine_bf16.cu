// Combination kernels that take the last chunk first, bf16 gradients, K = 1..3,
// fp32 or bf16 output.
#include "combine_impl.cuh"

namespace bkmoo {
static const void* const kCombineTable[combine_last_first_max_k(BKMOO_BF16)][2] = {
    BKMOO_COMBINE_ROW(1, BKMOO_BF16), BKMOO_COMBINE_ROW(2, BKMOO_BF16),
    BKMOO_COMBINE_ROW(3, BKMOO_BF16)};
const void* combine_fn_bf16(int K, int dtype_out) { return kCombineTable[K - 1][dtype_out]; }
}  // namespace bkmoo
