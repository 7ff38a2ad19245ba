// Combination kernels that take the last chunk first, fp32 gradients, K = 1..4
// (last_first_bytes in host.cu), fp32 or bf16 output.
#include "combine_impl.cuh"

namespace bkmoo {
static const void* const kFew[4][2] = {
    BKMOO_COMBINE_ROW(1, BKMOO_F32), BKMOO_COMBINE_ROW(2, BKMOO_F32),
    BKMOO_COMBINE_ROW(3, BKMOO_F32), BKMOO_COMBINE_ROW(4, BKMOO_F32)};
const void* combine_fn_f32(int K, int dtype_out) {
  return K <= 4 ? kFew[K - 1][dtype_out] : nullptr;
}
}  // namespace bkmoo
