// Combination kernels that take the last chunk first, bf16 gradients, K = 1..3
// and 12..16 (last_first_bytes in host.cu), fp32 or bf16 output.
#include "combine_impl.cuh"

namespace bkmoo {
static const void* const kFew[3][2] = {BKMOO_COMBINE_ROW(1, BKMOO_BF16),
                                       BKMOO_COMBINE_ROW(2, BKMOO_BF16),
                                       BKMOO_COMBINE_ROW(3, BKMOO_BF16)};
static const void* const kMany[5][2] = {
    BKMOO_COMBINE_ROW(12, BKMOO_BF16), BKMOO_COMBINE_ROW(13, BKMOO_BF16),
    BKMOO_COMBINE_ROW(14, BKMOO_BF16), BKMOO_COMBINE_ROW(15, BKMOO_BF16),
    BKMOO_COMBINE_ROW(16, BKMOO_BF16)};
const void* combine_fn_bf16(int K, int dtype_out) {
  return K <= 3 ? kFew[K - 1][dtype_out] : K >= 12 ? kMany[K - 12][dtype_out] : nullptr;
}
}  // namespace bkmoo
