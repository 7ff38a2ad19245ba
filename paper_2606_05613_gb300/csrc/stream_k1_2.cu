// Streamed resolve kernels, K = 1 and 2, fp32 / bf16 gradients.
#include "stream_resolve.cuh"

namespace bkmoo {
const void* stream_fn_k1_2(int K, int dti) {
  if (K == 1)
    return dti == BKMOO_F32 ? (const void*)stream_resolve_kernel<1, BKMOO_F32>
                            : (const void*)stream_resolve_kernel<1, BKMOO_BF16>;
  return dti == BKMOO_F32 ? (const void*)stream_resolve_kernel<2, BKMOO_F32>
                          : (const void*)stream_resolve_kernel<2, BKMOO_BF16>;
}
int stream_threads() { return 32 * kStreamWarps; }
int stream_smem(int K) { return stream_smem_bytes(K); }
int stream_stage_kib(int K) { return stream_stage_bytes(K) / 1024; }
int stream_chunk_stages(int K) { return kVecPerThread / stream_items(K); }
}  // namespace bkmoo
