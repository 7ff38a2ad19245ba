// Streamed resolve kernels, K = 5 and 6, fp32 / bf16 gradients.
#include "stream_resolve.cuh"

namespace bkmoo {
const void* stream_fn_k5_6(int K, int dti) {
  if (K == 5)
    return dti == BKMOO_F32 ? (const void*)stream_resolve_kernel<5, BKMOO_F32>
                            : (const void*)stream_resolve_kernel<5, BKMOO_BF16>;
  return dti == BKMOO_F32 ? (const void*)stream_resolve_kernel<6, BKMOO_F32>
                          : (const void*)stream_resolve_kernel<6, BKMOO_BF16>;
}
}  // namespace bkmoo
