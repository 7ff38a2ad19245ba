// Streamed resolve kernels, K = 3 and 4, fp32 / bf16 gradients.
#include "stream_resolve.cuh"

namespace bkmoo {
const void* stream_fn_k3_4(int K, int dti) {
  if (K == 3)
    return dti == BKMOO_F32 ? (const void*)stream_resolve_kernel<3, BKMOO_F32>
                            : (const void*)stream_resolve_kernel<3, BKMOO_BF16>;
  return dti == BKMOO_F32 ? (const void*)stream_resolve_kernel<4, BKMOO_F32>
                          : (const void*)stream_resolve_kernel<4, BKMOO_BF16>;
}
}  // namespace bkmoo
