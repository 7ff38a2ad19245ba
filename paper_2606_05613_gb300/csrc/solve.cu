// Solve pass: one warp, or one block of eight, per bucket.  It reduces the
// bucket's per-chunk Gram partials in a fixed order (fp64; sum_chunk_rows in
// common.cuh: sets of sixteen rows for K <= 8, eight interleaved sums) into G in
// shared memory; one warp solves the bucket's rule (solver.cuh) and writes beta
// and the bucket's status.
#include "solver.cuh"

namespace bkmoo {
namespace {

using namespace solver;

__global__ void __launch_bounds__(32 * kSolveWarpsPerBlock)
    solve_kernel(const PlanView v, const SolveParams p, float* out_weights,
                 int32_t* out_status) {
  __shared__ double Gs[kSolveWarpsPerBlock][kMaxK * kMaxK];
  __shared__ double Bs[kSolveWarpsPerBlock][kMaxK];
  __shared__ float Fs[kSolveWarpsPerBlock][kMaxK * kMaxK];
  grid_wait();
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int64_t b = v.b_lo + (int64_t)blockIdx.x * kSolveWarpsPerBlock + wi;
  if (b >= v.b_hi) return;
  const int K = v.K;
  if (!header_ok(v)) {
    if (lane == 0 && out_status) out_status[b] = BKMOO_ERR_WORKSPACE;
    return;
  }
  double* G = Gs[wi];
  double* beta = Bs[wi];
  reduce_bucket(v, b, G, lane);
  const int st = solve_bucket_warp<0>(K, G, Fs[wi], p, b, beta, lane);
  for (int k = lane; k < K; k += 32) {
    const float f = (float)beta[k];
    v.beta[b * K + k] = f;
    if (out_weights) out_weights[b * K + k] = f;
  }
  if (lane == 0 && out_status) out_status[b] = st;
}

// One block of eight warps per bucket (solve_wide, below): the warps share the
// rows, one solves.  One warp adds rows at one fp64 instruction per 64 cycles; a
// 400-chunk K = 4 bucket: 68 -> 60 us for the three launches of the bucket alone.
__global__ void __launch_bounds__(32 * kWideWarps)
    solve_wide_kernel(const PlanView v, const SolveParams p, float* out_weights,
                      int32_t* out_status) {
  __shared__ double t8[kWideWarps * tri(kMaxK)];
  __shared__ double G[kMaxK * kMaxK];
  __shared__ double beta[kMaxK];
  __shared__ float Gf[kMaxK * kMaxK];
  grid_wait();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t b = v.b_lo + blockIdx.x;
  const int K = v.K;
  if (!header_ok(v)) {
    if (threadIdx.x == 0 && out_status) out_status[b] = BKMOO_ERR_WORKSPACE;
    return;
  }
  reduce_bucket_wide(v, b, t8, lane, w);
  __syncthreads();
  if (w != 0) return;
  gram_from_sums(K, t8, G, lane);
  const int st = solve_bucket_warp<0>(K, G, Gf, p, b, beta, lane);
  for (int k = lane; k < K; k += 32) {
    const float f = (float)beta[k];
    v.beta[b * K + k] = f;
    if (out_weights) out_weights[b * K + k] = f;
  }
  if (lane == 0 && out_status) out_status[b] = st;
}

__global__ void __launch_bounds__(32 * kWideWarps)
    gram_finalize_wide_kernel(const PlanView v, double* out_gram) {
  __shared__ double t8[kWideWarps * tri(kMaxK)];
  __shared__ double G[kMaxK * kMaxK];
  grid_wait();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t b = blockIdx.x;
  if (!header_ok(v)) return;
  const int K = v.K;
  reduce_bucket_wide(v, b, t8, lane, w);
  __syncthreads();
  if (w != 0) return;
  gram_from_sums(K, t8, G, lane);
  for (int i = lane; i < K * K; i += 32) out_gram[b * K * K + i] = G[i];
}

__global__ void __launch_bounds__(32 * kSolveWarpsPerBlock)
    gram_finalize_kernel(const PlanView v, double* out_gram) {
  __shared__ double Gs[kSolveWarpsPerBlock][kMaxK * kMaxK];
  grid_wait();
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int64_t b = (int64_t)blockIdx.x * kSolveWarpsPerBlock + wi;
  if (b >= v.n_buckets) return;
  if (!header_ok(v)) return;
  const int K = v.K;
  double* G = Gs[wi];
  reduce_bucket(v, b, G, lane);
  for (int i = lane; i < K * K; i += 32) out_gram[b * K * K + i] = G[i];
}

// Block (x = group j, y = a stride of the buckets): of a bucket of more than
// kGroupMinChunks chunks, eight warps sum the rows of the chunks
// [c0 + 512 j, c0 + 512 (j+1)) (as sum_chunk_rows does) into the group's first
// row, which no other block reads.  Every warp looks 32 of the block's buckets
// over at a time, so a plan of many small buckets costs few blocks.  fp64 adds
// bound it, hence the eight warps.  Gram call with one warp a group and with
// eight: K = 4, one bucket of 1100 chunks 109 -> 67 us, one of 6000 281 -> 239, the
// same beside 1000 small buckets 317 -> 254; K = 16, 6000 chunks 1053 -> 973.
__global__ void __launch_bounds__(32 * kWideWarps) group_reduce_kernel(const PlanView v) {
  __shared__ double t8[kWideWarps * tri(kMaxK)];
  grid_wait();
  grid_release();
  if (!header_ok(v)) return;
  const int lane = threadIdx.x & 31, P = tri(v.K);
  for (int64_t b0 = v.b_lo + blockIdx.y; b0 < v.b_hi; b0 += 32 * (int64_t)gridDim.y) {
    const int64_t bl = b0 + lane * (int64_t)gridDim.y;
    unsigned large = __ballot_sync(
        0xffffffffu,
        bl < v.b_hi && v.chunk_prefix[bl + 1] - v.chunk_prefix[bl] > kGroupMinChunks);
    for (; large; large &= large - 1) {
      const int64_t b = b0 + (__ffs(large) - 1) * (int64_t)gridDim.y;
      const int64_t c0 = v.chunk_prefix[b] + (int64_t)blockIdx.x * kGroupChunks;
      const int64_t left = v.chunk_prefix[b + 1] - c0;
      if (left <= 0) continue;
      double* row = v.partials + c0 * P;
      sum_rows_wide(row, P, min(kGroupChunks, left), P, v.K <= kStreamMaxK, t8, lane,
                    threadIdx.x >> 5);
      __syncthreads();
      for (int p = threadIdx.x; p < P; p += blockDim.x) row[p] = tree8_entry(t8, P, p);
      __syncthreads();
    }
  }
}

// Element i of the fp64 division / square-root helpers of the fast solvers
// (op 0: a[i] / b[i] by div_nr, op 1: sqrt(a[i]) by sqrt_nr); grid-stride.
__global__ void selftest_fp64_kernel(int op, const double* a, const double* b, double* out,
                                     int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = op == 0 ? div_nr(a[i], b[i]) : sqrt_nr(a[i]);
}

}  // namespace

cudaError_t launch_selftest_fp64(int op, const double* a, const double* b, double* out, int64_t n,
                                 cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  int64_t grid = (n + 255) / 256;
  if (grid > 4096) grid = 4096;
  selftest_fp64_kernel<<<(unsigned)grid, 256, 0, s>>>(op, a, b, out, n);
  return cudaGetLastError();
}

// Blocks of the pre-reduction: seven per SM.
constexpr int64_t kGroupBlocks = 1024;

cudaError_t launch_group_reduce(const PlanView& v, cudaStream_t s, bool behind) {
  if (v.max_chunks <= kGroupMinChunks || v.b_hi <= v.b_lo) return cudaSuccess;
  const int64_t gx = (v.max_chunks + kGroupChunks - 1) / kGroupChunks;
  int64_t gy = v.b_hi - v.b_lo;
  if (gx * gy > kGroupBlocks) gy = kGroupBlocks / gx > 0 ? kGroupBlocks / gx : 1;
  PlanView va = v;
  void* args[] = {&va};
  return launch_behind((const void*)group_reduce_kernel, dim3((unsigned)gx, (unsigned)gy),
                       dim3(32 * kWideWarps), args, 0, s, behind);
}

// Whether a window's buckets take a block of eight warps each; otherwise a warp
// each, four to a block, in a plain launch.  Launched behind the Gram pass, the
// four-warp blocks gather on the few SMs that finish first and share their fp64
// units: 608 buckets, K = 4, Frank-Wolfe alone 631 us behind, 293 plain, 489 with
// a block a bucket; CAGrad, small buckets: 45, 35, 40.  A block a bucket, behind,
// wins up to two buckets per SM (304, CAGrad: 28 against 42 and 31) and, by 0.04
// us for each row of the longest bucket against 0.02 for each bucket, where that
// bucket is long (1000 buckets of 300 elements beside one of 1000 chunks, K = 4:
// 169 against 182, 2000 beside one of 400 147 against 116).
static cudaError_t solve_wide(const PlanView& v, int64_t nb, bool* wide, int* sms) {
  const cudaError_t e = sm_count(sms);
  const int64_t rows = v.max_chunks > kGroupMinChunks
                           ? (v.max_chunks + kGroupChunks - 1) / kGroupChunks
                           : v.max_chunks;
  *wide = nb <= 2 * (int64_t)*sms || 2 * rows >= nb;
  return e;
}

cudaError_t launch_solve(const PlanView& v, const SolveParams& p, float* out_weights,
                         int32_t* out_status, cudaStream_t s, bool behind) {
  const int64_t nb = v.b_hi - v.b_lo;
  if (nb <= 0) return cudaSuccess;
  bool wide = false;
  int sms = 0;
  const cudaError_t e = solve_wide(v, nb, &wide, &sms);
  if (e != cudaSuccess) return e;
  // A few us of solve on every SM: more than six buckets per SM by exact MGDA (1024
  // buckets of 4099 elements, plain / behind: K = 4 52.6 / 47.1 us, K = 5 66.9 / 54.9;
  // PCGrad 56.9 / 55.5 and 69.2 / 65.8, but K = 8 109.7 / 126.2, its MGDA 97.5 / 99.3,
  // and K = 2 CAGrad 43.4 / 50.2; 608 buckets, MGDA, K = 4 28.7 / 30.0).
  const bool many_short = p.rule == BKMOO_MGDA && (p.flags & BKMOO_FLAG_POLISH) && v.K < 8 &&
                          nb > 6 * (int64_t)sms;
  const int64_t grid = wide ? nb : (nb + kSolveWarpsPerBlock - 1) / kSolveWarpsPerBlock;
  PlanView va = v;
  SolveParams pa = p;
  void* args[] = {&va, &pa, &out_weights, &out_status};
  return launch_behind(wide ? (const void*)solve_wide_kernel : (const void*)solve_kernel,
                       dim3((unsigned)grid),
                       dim3(32 * (wide ? kWideWarps : kSolveWarpsPerBlock)), args, 0, s,
                       behind && (wide || many_short));
}

cudaError_t launch_gram_finalize(const PlanView& v, double* out_gram, cudaStream_t s,
                                 bool behind) {
  const int64_t nb = v.n_buckets;
  if (nb == 0) return cudaSuccess;
  bool wide = false;
  int sms = 0;
  const cudaError_t e = solve_wide(v, nb, &wide, &sms);
  if (e != cudaSuccess) return e;
  const int64_t grid = wide ? nb : (nb + kSolveWarpsPerBlock - 1) / kSolveWarpsPerBlock;
  PlanView va = v;
  void* args[] = {&va, &out_gram};
  return launch_behind(wide ? (const void*)gram_finalize_wide_kernel
                            : (const void*)gram_finalize_kernel,
                       dim3((unsigned)grid),
                       dim3(32 * (wide ? kWideWarps : kSolveWarpsPerBlock)), args, 0, s,
                       behind && wide);
}

}  // namespace bkmoo
