// Streamed resolve kernels, K = 7 and 8, fp32 / bf16 gradients.
#include "stream_resolve.cuh"

namespace bkmoo {
const void* stream_fn_k7_8(int K, int dti) {
  if (K == 7)
    return dti == BKMOO_F32 ? (const void*)stream_resolve_kernel<7, BKMOO_F32>
                            : (const void*)stream_resolve_kernel<7, BKMOO_BF16>;
  return dti == BKMOO_F32 ? (const void*)stream_resolve_kernel<8, BKMOO_F32>
                          : (const void*)stream_resolve_kernel<8, BKMOO_BF16>;
}
}  // namespace bkmoo
