// Kernel tables and launchers that launch nothing and note what they were asked
// for (see fake_runtime.cpp).
#include "common.cuh"

extern char kGram, kPrefetchGram, kBulkGram, kLastFirst, kPrefetch, kStream;
void note(const char* what);

namespace bkmoo {
const void* gram_partials_fn_f32(int) { return &kGram; }
const void* gram_partials_fn_bf16(int) { return &kGram; }
const void* gram_prefetch_fn(int, int) { return &kPrefetchGram; }
int gram_prefetch_smem(int) { return 1; }
int gram_prefetch_min_k() { return 12; }
const void* gram_bulk_fn(int K, int) { return K >= kBulkMinK && K <= kBulkMaxK ? &kBulkGram : nullptr; }
int gram_bulk_smem(int) { return 1; }
int gram_bulk_threads() { return 288; }
const void* combine_prefetch_fn(int, int, int) { return &kPrefetch; }
int combine_prefetch_smem(int) { return 1; }
const void* combine_fn_f32(int, int) { return &kLastFirst; }
const void* combine_fn_bf16(int, int) { return &kLastFirst; }
const void* stream_fn_k1_2(int, int) { return &kStream; }
const void* stream_fn_k3_4(int, int) { return &kStream; }
const void* stream_fn_k5_6(int, int) { return &kStream; }
const void* stream_fn_k7_8(int, int) { return &kStream; }
int stream_threads() { return 512; }
int stream_smem(int) { return 1; }
int stream_stage_kib(int) { return 32; }
int stream_chunk_stages(int) { return 8; }
cudaError_t launch_solve(const PlanView&, const SolveParams&, float*, int32_t*, cudaStream_t, bool) {
  note("solve");
  return cudaSuccess;
}
cudaError_t launch_gram_finalize(const PlanView&, double*, cudaStream_t, bool) {
  note("finalize");
  return cudaSuccess;
}
cudaError_t launch_selftest_fp64(int, const double*, const double*, double*, int64_t, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t launch_group_reduce(const PlanView& v, cudaStream_t, bool) {
  if (v.max_chunks > kGroupMinChunks) note("groups");
  return cudaSuccess;
}
}  // namespace bkmoo
