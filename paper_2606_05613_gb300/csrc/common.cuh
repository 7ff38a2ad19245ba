// Internal definitions shared by the translation units of the bkmoo CUDA
// library: workspace layout, kernel argument blocks, 16-byte vector access
// and the chunk -> bucket lookup.  Not part of the C ABI (include/bkmoo.h).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "bkmoo.h"

namespace bkmoo {

constexpr int kMaxK = 16;
// Largest K of the streamed kernel (stream_resolve.cuh).
constexpr int kStreamMaxK = 8;
constexpr int kThreads = 256;              // CTA size of the streaming kernels
constexpr int kWarps = kThreads / 32;
constexpr int kVecPerThread = 16;          // 16-byte vectors per thread per Gram chunk
constexpr uint32_t kMagic = 0x4f4d4b42u;   // "BKMO"
constexpr int kSolveWarpsPerBlock = 4;
// A bucket with more than kGroupMinChunks chunks has its chunk partials
// pre-reduced in groups of kGroupChunks (group_reduce_kernel, solve.cu)
// before the per-bucket reduction reads them: one warp would otherwise read
// every partial of a huge bucket (the one-bucket "global" variant) alone.
constexpr int64_t kGroupChunks = 512;
constexpr int64_t kGroupMinChunks = 1024;

// Chunk rows are summed in sets of kSetChunks (K <= kStreamMaxK).
constexpr int kSetChunks = 16;

__host__ __device__ constexpr int tri(int K) { return K * (K + 1) / 2; }
__host__ __device__ constexpr int elems_per_vec(int dtype) { return dtype == BKMOO_F32 ? 4 : 8; }
__host__ __device__ constexpr int64_t chunk_elems(int dtype) {
  return (int64_t)kThreads * kVecPerThread * elems_per_vec(dtype);
}

// First 256 bytes of every workspace.
struct WsHeader {
  uint32_t magic;
  int32_t K;
  int32_t in_dtype;
  int32_t status;        // device-side error word: BKMOO_OK or the first error
  int64_t n_buckets;
  int64_t n_elems;
  int64_t n_chunks;
  int64_t chunk_elems;
  uint64_t plan_hash;
  int64_t reserved[25];
};
static_assert(sizeof(WsHeader) == 256, "header is one 256-byte block");

// Byte offsets of the workspace regions (identical on host and device).
struct WsLayout {
  size_t offsets;        // int64 [B + 1]   bucket boundaries (elements)
  size_t chunk_prefix;   // int64 [B + 1]   first Gram chunk of each bucket
  size_t partials;       // double [n_chunks][P] per-chunk Gram partials
  size_t beta;           // float [B][K]    coefficients of the last resolve
  size_t total;          // end of the regions above
  // streamed path only
  size_t rows;           // uint64 [n_chunks][stream_row_words(K)], K <= kStreamMaxK
  size_t chunk_bucket;   // int32 [n_chunks] bucket of each chunk
  size_t total_all;
};

__host__ __device__ inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Host-side plan helpers shared by every entry point.
// Offsets start at 0 and increase strictly (no empty bucket).
inline bool offsets_ok(const int64_t* off, int64_t B) {
  if (!off || B < 0 || off[0] != 0) return false;
  for (int64_t b = 0; b < B; ++b)
    if (off[b + 1] <= off[b]) return false;
  return true;
}

// Gram chunks of a plan: each bucket is cut into chunks of ch elements, the
// last one short.
inline int64_t count_chunks(const int64_t* off, int64_t B, int64_t ch) {
  int64_t n = 0;
  for (int64_t b = 0; b < B; ++b) n += (off[b + 1] - off[b] + ch - 1) / ch;
  return n;
}

// FNV-1a over the 64-bit words that define a plan (K, dtype, B, offsets);
// kept in the workspace header and checked by every kernel.
inline uint64_t plan_hash(int32_t K, int32_t dt, const int64_t* off, int64_t B) {
  uint64_t h = 0xcbf29ce484222325ull;
  auto mix = [&h](uint64_t x) {
    h ^= x;
    h *= 0x100000001b3ull;
  };
  mix((uint64_t)K);
  mix((uint64_t)dt);
  mix((uint64_t)B);
  for (int64_t b = 0; b <= B; ++b) mix((uint64_t)off[b]);
  return h;
}

__host__ __device__ inline WsLayout ws_layout(int K, int64_t B, int64_t n_chunks) {
  WsLayout L;
  size_t at = sizeof(WsHeader);
  L.offsets = at;
  at = align256(at + sizeof(int64_t) * (size_t)(B + 1));
  L.chunk_prefix = at;
  at = align256(at + sizeof(int64_t) * (size_t)(B + 1));
  L.partials = at;
  at = align256(at + sizeof(double) * (size_t)n_chunks * (size_t)tri(K));
  L.beta = at;
  at = align256(at + sizeof(float) * (size_t)B * (size_t)K);
  L.total = at;
  L.rows = at;
  if (K <= kStreamMaxK)
    at = align256(at + sizeof(uint64_t) * (size_t)n_chunks * (size_t)(tri(K) + K + 1));
  L.chunk_bucket = at;
  at = align256(at + sizeof(int32_t) * (size_t)n_chunks);
  L.total_all = at;
  return L;
}

struct GradPtrs {
  const void* p[kMaxK];
};

// Everything a kernel needs to find its data.
struct PlanView {
  WsHeader* hdr;
  const int64_t* offsets;
  const int64_t* chunk_prefix;
  double* partials;
  float* beta;
  int64_t n_buckets;
  int64_t n_chunks;
  int64_t chunk_elems;
  uint64_t plan_hash;
  int32_t K;
  int32_t in_dtype;
  // The part of the plan one launch works on: chunks [c_lo, c_hi) of buckets
  // [b_lo, b_hi) (the whole plan except in the windowed host-memory path).
  int64_t c_lo, c_hi;
  int64_t b_lo, b_hi;
  int64_t elems;        // elements of one language in [b_lo, b_hi) (host-computed)
  int64_t max_chunks;   // most chunks in one bucket of the plan (host-computed)
};

// Whole-plan window of a view whose n_buckets and n_chunks are set.
__host__ __device__ inline void full_window(PlanView& v) {
  v.c_lo = 0;
  v.c_hi = v.n_chunks;
  v.b_lo = 0;
  v.b_hi = v.n_buckets;
}

// The streamed path's view (stream_resolve.cuh): the plan's window plus one
// row of 64-bit words per chunk:
//   [0, P)       the chunk's partials,
//   [P, P + K)   in a bucket's first chunk: the bucket's coefficients,
//   [P + K]      in the window's first row: the give-up flag.
// Every word is 0 until it is written (see st_row and st_beta).
struct StreamView {
  PlanView v;
  uint64_t* rows;               // row of chunk w0
  const int32_t* chunk_bucket;  // bucket of every chunk of the plan
  int32_t* give_up;             // set once a wait for another CTA ran out
  int64_t w0;                   // first chunk of the window
  int32_t lead;                 // stages the Gram may run ahead of the combination
  int32_t l2_stages;            // stages a CTA asks L2 to keep
  int32_t n_stream;             // CTAs that stream (chunk w0 + i by CTA i mod n_stream); the
                                // others solve
  int32_t team;                 // warps of a solver CTA that share a bucket: 2, 4 or 8
  int32_t reset;                // clear the workspace status word first
};
__host__ __device__ constexpr int stream_row_words(int K) { return tri(K) + K + 1; }

struct SolveParams {
  int32_t rule;
  int32_t max_iter;
  double tol;
  double cagrad_c;
  uint64_t seed;
  uint64_t step;
  uint32_t flags;
};

// Launch that may begin before the kernel ahead of it in the stream has ended
// (programmatic dependent launch): its CTAs are in place when that kernel's
// last one leaves, instead of 2-4 us later.  Every kernel launched so waits at
// its top (grid_wait) for that kernel's end, so an end implies the ends of all
// before it.
inline cudaError_t launch_behind(const void* fn, dim3 grid, dim3 block, void** args, size_t smem,
                                 cudaStream_t s, bool behind) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = behind ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// ---------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------

// Until the kernels ahead in the stream have ended and their writes are
// visible (nothing to wait for after a plain launch).
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// From here on the next kernel's CTAs may be put beside this kernel's.
__device__ __forceinline__ void grid_release() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ bool header_ok(const PlanView& v) {
  const WsHeader* h = v.hdr;
  return h->magic == kMagic && h->plan_hash == v.plan_hash && h->K == v.K &&
         h->in_dtype == v.in_dtype && h->n_buckets == v.n_buckets &&
         h->n_chunks == v.n_chunks;
}

__device__ __forceinline__ void record_error(WsHeader* h, int code) {
  atomicCAS(&h->status, 0, code);
}

// Fixed order of the fp64 sums over Gram rows, one entry per thread (rows
// rs doubles apart): eight interleaved sums (row c into sum c mod 8), then a
// fixed tree.
__device__ __forceinline__ double tree8(const double (&t)[8]) {
  return ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
}
__device__ __forceinline__ double sum_rows8(const double* src, int64_t rs, int64_t n) {
  double t[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int64_t c = 0;
  for (; c + 8 <= n; c += 8, src += 8 * rs) {
#pragma unroll
    for (int j = 0; j < 8; ++j) t[j] += src[j * rs];
  }
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (c + j < n) t[j] += src[j * rs];
  return tree8(t);
}
// A set: the first kSetChunks (or all left) of `left` rows, a whole one in
// one round trip.  (No partial is -0, so adding the first eight to 0, as
// sum_rows8 does, would change nothing.)
__device__ __forceinline__ double set_sum(const double* row, int64_t rs, int64_t left) {
  if (left < kSetChunks) return sum_rows8(row, rs, left);
  double x[kSetChunks], u[8];
#pragma unroll
  for (int i = 0; i < kSetChunks; ++i) x[i] = row[i * rs];
#pragma unroll
  for (int i = 0; i < 8; ++i) u[i] = x[i] + x[i + 8];
  return tree8(u);
}
// Chunk rows: for K <= kStreamMaxK sets of kSetChunks rows, then the sets'
// sums in the same way -- the order in which the streamed kernel, whose sets
// are summed by different warps of a team, arrives at them.
__device__ __forceinline__ double sum_chunk_rows(const double* src, int64_t rs, int64_t n, int K) {
  if (n == 1) return *src;              // (adding zeros changes no partial)
  if (K > kStreamMaxK) return sum_rows8(src, rs, n);
  if (n <= kSetChunks) return set_sum(src, rs, n);
  double t[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int64_t c = 0; c < n; c += 8 * kSetChunks) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int64_t at = c + j * kSetChunks;
      if (at < n) t[j] += set_sum(src + at * rs, rs, n - at);
    }
  }
  return tree8(t);
}

// Bucket b with chunk_prefix[b] <= w < chunk_prefix[b+1]; `hint` is tried
// first (chunks of one CTA increase monotonically).
__device__ __forceinline__ int64_t find_bucket(const int64_t* cp, int64_t B, int64_t w,
                                               int64_t hint) {
  if (hint < B && cp[hint] <= w && w < cp[hint + 1]) return hint;
  if (hint + 1 < B && cp[hint + 1] <= w && w < cp[hint + 2]) return hint + 1;
  int64_t lo = 0, hi = B;
  while (hi - lo > 1) {
    int64_t mid = (lo + hi) >> 1;
    if (cp[mid] <= w) lo = mid;
    else hi = mid;
  }
  return lo;
}

// 16-byte loads.  `nc`: read-only path, no L1 allocation (streams that are
// read once by this kernel).  `cs`: coherent, evict-first (combine, which
// may write in place over one of the inputs).
__device__ __forceinline__ uint4 ld16_nc(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}
__device__ __forceinline__ uint4 ld16_cs(const void* p) {
  uint4 r;
  asm volatile("ld.global.cs.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}
__device__ __forceinline__ void st16_cs(void* p, uint4 v) {
  asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ void st8_cs(void* p, uint2 v) {
  asm volatile("st.global.cs.v2.u32 [%0], {%1,%2};" ::"l"(p), "r"(v.x), "r"(v.y) : "memory");
}

__device__ __forceinline__ uint32_t word(const uint4& r, int i) {
  return i == 0 ? r.x : i == 1 ? r.y : i == 2 ? r.z : r.w;
}

// Element e of a 16-byte vector as fp32 (bf16 widened exactly).
template <int DT>
__device__ __forceinline__ float vec_elem(const uint4& r, int e) {
  if (DT == BKMOO_F32) return __uint_as_float(word(r, e));
  const uint32_t w = word(r, e >> 1);
  return (e & 1) ? __uint_as_float(w & 0xffff0000u) : __uint_as_float(w << 16);
}

template <int DT>
__device__ __forceinline__ float load_scalar(const void* base, int64_t i) {
  if (DT == BKMOO_F32) return static_cast<const float*>(base)[i];
  const uint16_t h = static_cast<const uint16_t*>(base)[i];
  return __uint_as_float((uint32_t)h << 16);
}

// ---------------------------------------------------------------------------
// Kernel tables and launchers
// ---------------------------------------------------------------------------

// Gram-pass kernels, signature (GradPtrs, PlanView); gram_f32.cu / gram_bf16.cu.
const void* gram_partials_fn_f32(int K);
const void* gram_partials_fn_bf16(int K);

// Gram-pass kernels with a per-thread shared-memory prefetch (same signature,
// kThreads threads, gram_prefetch_smem(K) bytes of dynamic shared memory) for
// K >= gram_prefetch_min_k(); nullptr below; gram_prefetch.cu.
const void* gram_prefetch_fn(int K, int dt);
int gram_prefetch_smem(int K);
int gram_prefetch_min_k();

// Gram-pass kernels fed by bulk copies (same signature, gram_bulk_threads()
// threads, gram_bulk_smem(K) bytes of dynamic shared memory), K = kBulkMinK ..
// kBulkMaxK, nullptr outside; gram_bulk.cu.
constexpr int kBulkMinK = 2, kBulkMaxK = 8;
const void* gram_bulk_fn(int K, int dt);
int gram_bulk_smem(int K);
int gram_bulk_threads();

// Combine kernels with a per-thread shared-memory prefetch (same signature,
// combine_prefetch_smem(K) bytes of dynamic shared memory), every K;
// combine_prefetch.cu, combine_prefetch_k9_16.cu.
const void* combine_prefetch_fn(int K, int dti, int dto);
const void* combine_prefetch_fn_k9_16(int K, int dti, int dto);
int combine_prefetch_smem(int K);

// Combine kernels that take the last chunk first, for short windows and short
// chunks (last_first_bytes in host.cu), signature (GradPtrs, PlanView, void* out);
// combine_*.cu.
const void* combine_fn_f32(int K, int dtype_out);
const void* combine_fn_bf16(int K, int dtype_out);

// Streamed resolve kernels (stream_*.cu), K <= kStreamMaxK, signature
// (GradPtrs, StreamView, SolveParams, float* out_weights, int32_t* out_status,
// void* out, int dtype_out), stream_threads() threads and stream_smem(K) bytes
// of dynamic shared memory, one CTA per SM, co-resident.
const void* stream_fn_k1_2(int K, int dti);
const void* stream_fn_k3_4(int K, int dti);
const void* stream_fn_k5_6(int K, int dti);
const void* stream_fn_k7_8(int K, int dti);
int stream_threads();
int stream_smem(int K);
int stream_stage_kib(int K);
int stream_chunk_stages(int K);   // stages of a whole chunk

// SMs of the current device (cached; host.cu).
cudaError_t sm_count(int* n);

// solve.cu
// `behind`: launched behind the Gram pass (launch_behind).
cudaError_t launch_solve(const PlanView& v, const SolveParams& p, float* out_weights,
                         int32_t* out_status, cudaStream_t s, bool behind);
cudaError_t launch_gram_finalize(const PlanView& v, double* out_gram, cudaStream_t s, bool behind);
// The fp64 division / square-root helpers of the fast solvers, element-wise
// (self-test of their accuracy against the correctly rounded operations).
cudaError_t launch_selftest_fp64(int op, const double* a, const double* b, double* out, int64_t n,
                                 cudaStream_t s);
// After a Gram pass over the view's window: the group pre-reduction of its
// large buckets (a no-op when no bucket has more than kGroupMinChunks chunks).
cudaError_t launch_group_reduce(const PlanView& v, cudaStream_t s, bool behind);

}  // namespace bkmoo
