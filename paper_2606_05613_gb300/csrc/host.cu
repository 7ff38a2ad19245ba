// Host side of the C ABI (include/bkmoo.h): argument checks, the bucket plan,
// the workspace image, the launch sequence Gram -> solve -> combine on the
// caller's stream (whole plan, a bucket range, or windows of buckets staged
// from host memory), and the streamed launch.  Nothing here
// allocates device memory (the host path creates two copy streams and a few
// events per call).
#include <cuda_runtime.h>

#include <cstring>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

#include "common.cuh"

using namespace bkmoo;

namespace {

constexpr int32_t kVersion = 200;  // 0.2.0: bucket-range and host-memory entry points

bool dtype_ok(int32_t dt) { return dt == BKMOO_F32 || dt == BKMOO_BF16; }
int elem_bytes(int32_t dt) { return dt == BKMOO_F32 ? 4 : 2; }
bool aligned(const void* p, uintptr_t a) { return ((uintptr_t)p & (a - 1)) == 0; }

struct LaunchCache {
  std::mutex mu;
  std::map<int, int> sms;
  std::map<std::pair<int, const void*>, int> occ;
};
LaunchCache& cache() {
  static LaunchCache c;
  return c;
}

// With the cache's lock held.
cudaError_t device_sms(LaunchCache& c, int dev, int* n) {
  auto it = c.sms.find(dev);
  if (it == c.sms.end()) {
    const cudaError_t e = cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    it = c.sms.emplace(dev, *n).first;
  }
  *n = it->second;
  return cudaSuccess;
}

// Resident CTAs of `fn` on the current device times its SM count.  A kernel
// with dynamic shared memory gets its limit raised to that size once (the
// default limit of 48 KiB counts static and dynamic shared memory together).
cudaError_t persistent_grid(const void* fn, int threads, int* grid, int dyn_smem = 0) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  LaunchCache& c = cache();
  std::lock_guard<std::mutex> lk(c.mu);
  int sms = 0;
  e = device_sms(c, dev, &sms);
  if (e != cudaSuccess) return e;
  auto key = std::make_pair(dev, fn);
  auto jt = c.occ.find(key);
  if (jt == c.occ.end()) {
    int n = 0;
    if (dyn_smem > 0) {
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_smem);
      if (e != cudaSuccess) return e;
    }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, dyn_smem);
    if (e != cudaSuccess) return e;
    jt = c.occ.emplace(key, n < 1 ? 1 : n).first;
  }
  *grid = sms * jt->second;
  return cudaSuccess;
}

const void* gram_fn(int K, int dt) {
  return dt == BKMOO_F32 ? gram_partials_fn_f32(K) : gram_partials_fn_bf16(K);
}
const void* combine_fn(int K, int dti, int dto) {
  return dti == BKMOO_F32 ? combine_fn_f32(K, dto) : combine_fn_bf16(K, dto);
}
const void* stream_fn(int K, int dt) {
  return K <= 2 ? stream_fn_k1_2(K, dt)
                : (K <= 4 ? stream_fn_k3_4(K, dt)
                          : (K <= 6 ? stream_fn_k5_6(K, dt) : stream_fn_k7_8(K, dt)));
}

// Whether the streamed launch is the faster one for a window (both give the
// same results).  Measured on GB300 against the three launches on inputs not in
// L2 before: K = 1..8 fp32 and 2, 4, 5, 6, 8 bf16, MGDA, PCGrad and CAGrad, 1 to
// 4096 equal buckets of 16 KiB to 100 MiB a language, up to 3.3 GB of gradients.
// It reads the gradients little more than once and wins wherever the SMs' time
// goes into streaming; it loses where it goes into solves, which it does on the
// few SMs it sets aside.  Where it is taken it is at most 5 % behind, mostly 1.1
// to 1.6 times as fast.  The lines (streamed / three, us, fp32):
//  - K <= 4, more than 64 buckets: 0.5 MiB of gradients a bucket.  K = 4, 4096 of
//    0.5 MiB MGDA 445 / 724, CAGrad 535 / 754; 4096 of 0.25 MiB 248 / 386, but CAGrad
//    452 / 417; 1024 of 64 KiB 69 / 47, 129 / 55.  64 buckets of 64 KiB, CAGrad:
//    26 / 25.
//  - K >= 5, whose solves take 10-20 us: 96 MiB in all.  K = 8, 8 buckets of 4 MiB
//    MGDA 38.5 / 35.6, PCGrad 52.6 / 46.2; 16 of 4 MiB 40.2 / 47.2, 54.5 / 59.6; 64
//    of 2 MiB 54.6 / 66.8, 68.2 / 78.1.
//  - K >= 5: 1 MiB a bucket.  K = 8, 256 of 0.5 MiB MGDA 65.7 / 69.7, PCGrad 106 /
//    80; 128 of 1 MiB 54.9 / 68.3, 81.8 / 79.3; 256 of 1 MiB 84 / 113, 105 / 123.
//  - K >= 5, little of a bucket stays on the chip: more than 8 buckets only below
//    128 MiB each.  K = 5, 16 of 125 MiB MGDA 603 / 672, CAGrad 658 / 684; K = 6, 16
//    of 150 MiB 743 / 799, 812 / 813; K = 8 bf16, 16 of 200 MiB 974 / 1037, 1049 /
//    1049 (1100 / 1060 with an opposed language), 134 of 200 MiB 5967 / 5909; 8
//    of 200 MiB 489 / 534, 519 / 547.
//  - enormous buckets, of which nearly everything is read twice (ms): K >= 3 from
//    1 GiB each (K = 4 0.8 GiB 4.96 / 4.98, 1.6 GiB 5.01 / 4.98, 4 GB 5.10 / 5.04, one
//    of 65.5 GB 20.66 / 20.61; K = 3 1.2 GiB 3.91 / 3.87; K = 5 1 GiB 2.47 / 2.46; K = 8
//    0.8 GiB 1.89 / 1.92, one of 20 GB 6.15 / 5.92); K <= 2, whose second read costs
//    less, from 32 GiB (K = 2 4 GB 2.81 / 2.90; K = 1 the same within 1 %).
bool stream_wins(const PlanView& v) {
  if (v.K > kStreamMaxK || v.c_hi <= v.c_lo) return false;
  const int64_t nb = v.b_hi - v.b_lo;
  const double bytes = (double)v.elems * v.K * elem_bytes(v.in_dtype);
  const double mib = 1024.0 * 1024.0;
  if (v.K >= 5)
    return bytes >= 96.0 * mib && bytes >= 1.0 * mib * nb &&
           bytes < (nb <= 8 ? 1024.0 : 128.0) * mib * nb;
  if (bytes >= (v.K <= 2 ? 32768.0 : 1024.0) * mib * nb) return false;
  return nb <= 64 || bytes >= 0.5 * mib * nb;
}

// How a window is spread over the SMs, and how far the Gram may run ahead of
// the combination.
struct StreamShape {
  int n_stream, n_solve, team, lead_kib;
};
StreamShape stream_shape(const PlanView& v, int rule, int sms) {
  // From a bucket's last partial to its coefficients on every SM (us), from
  // globaltimer stamps under load (K = 2, 4, 8; K = 5..7 lie on the line between)
  // and, for K <= 4, the lead at which 1 and 4 MiB buckets run fastest.
  const double k4 = v.K < 4 ? v.K : 4, more = v.K > 4 ? v.K - 4 : 0;
  const double chain = rule == BKMOO_CAGRAD   ? 8 + 2 * k4 + 6 * more
                       : rule == BKMOO_PCGRAD ? 1 + 2.25 * k4 + 9 * more
                                              : 1.3 + 1.8 * k4 + 5.5 * more;
  const int64_t nb = v.b_hi - v.b_lo, nch = v.c_hi - v.c_lo;
  const int64_t sets = (v.max_chunks + kSetChunks - 1) / kSetChunks;
  StreamShape s;
  // a team's warps share a bucket's sets; at least two of the CTA's 16 warps,
  // so that no more than two solve on one scheduler
  s.team = sets <= 2 ? 2 : sets <= 4 ? 4 : 8;
  // teams: twice the buckets that complete during one chain
  const double period = (double)nch * v.chunk_elems * v.K * elem_bytes(v.in_dtype) / 7e6 / nb;
  double teams = 2.0 * chain / period + 1.0;
  if (teams > nb) teams = (double)nb;
  int64_t n = (int64_t)((teams * s.team + 15.0) / 16.0);
  if (n > sms / 10) n = sms / 10;
  // a small plan leaves SMs free: four solving warps on each
  const int64_t idle = sms - nch, want = (nb + 3) / 4;
  if (idle > n && want > n) n = want < idle ? want : idle;
  s.n_solve = n < 1 ? 1 : (int)n;
  s.n_stream = sms - s.n_solve;
  if (s.n_stream > nch) s.n_stream = (int)nch;
  // the copies in flight, a chunk, and what the Gram streams during the chain
  // (about 30 KiB per SM and us).  Less and the Gram stands still for the
  // chain, more and less of the window is kept (2.4 GB fp32 in 4 MiB buckets,
  // MGDA, us: K = 2 at 350 KiB 547, 400 534, 496 573; K = 3 460 590, 510 529, 640
  // 559; K = 4 570 559, 624 544), and for buckets of more than a chunk per SM,
  // which complete in waves of chunks, part of a chunk more (8 Qwen3-8B layers,
  // K = 4: 624 KiB 3353, 800 3288, 1200 3391)
  s.lead_kib = (int)(64 * v.K + 128 + 30 * chain);
  if (nch > nb * sms) s.lead_kib += 44 * v.K;
  return s;
}

// The streamed path over the view's window; *taken = false when the device
// cannot hold it (the caller then runs the three launches).
int launch_stream(const GradPtrs& g, const PlanView& v, const SolveParams& sp, void* ws,
                  float* out_weights, int32_t* out_status, void* out, int dto, bool reset,
                  bool* taken, cudaStream_t s) {
  *taken = false;
  const int64_t nch = v.c_hi - v.c_lo;
  if (v.K > kStreamMaxK || nch <= 0) return BKMOO_OK;
  const void* fn = stream_fn(v.K, v.in_dtype);
  const int smem = stream_smem(v.K);
  int sms = 0;
  if (persistent_grid(fn, stream_threads(), &sms, smem) != cudaSuccess) return BKMOO_ERR_CUDA;
  if (sms < 2) return BKMOO_OK;
  const StreamShape sh = stream_shape(v, sp.rule, sms);
  const WsLayout L = ws_layout(v.K, v.n_buckets, v.n_chunks);
  char* base = static_cast<char*>(ws);
  const size_t rw = (size_t)stream_row_words(v.K);
  StreamView sv;
  sv.v = v;
  sv.w0 = v.c_lo;
  sv.rows = reinterpret_cast<uint64_t*>(base + L.rows) + (size_t)v.c_lo * rw;
  sv.chunk_bucket = reinterpret_cast<const int32_t*>(base + L.chunk_bucket);
  sv.give_up = reinterpret_cast<int32_t*>(sv.rows + rw - 1);
  const int kib = stream_stage_kib(v.K);
  sv.n_stream = sh.n_stream;
  sv.team = sh.team;
  // (never less than a chunk and a stage: the combination of a chunk starts
  // after its Gram)
  const int least = stream_chunk_stages(v.K) + 1;
  sv.lead = sh.lead_kib / kib > least ? sh.lead_kib / kib : least;
  // 48-58 MB of L2 in all, what the re-read still finds there (K = 4, 1 MiB
  // buckets: 256 KiB per SM 871, 320 841, 384 818 us; more finds no more)
  sv.l2_stages = (v.K <= 4 ? 384 : 320) / kib;
  sv.reset = reset ? 1 : 0;
  if (cudaMemsetAsync(sv.rows, 0, (size_t)nch * rw * sizeof(uint64_t), s) != cudaSuccess)
    return BKMOO_ERR_CUDA;
  GradPtrs ga = g;
  SolveParams spa = sp;
  float* ow = out_weights;
  int32_t* os = out_status;
  void* outp = out;
  int d = dto;
  void* args[] = {&ga, &sv, &spa, &ow, &os, &outp, &d};
  const cudaError_t e =
      cudaLaunchCooperativeKernel(fn, dim3(sh.n_stream + sh.n_solve), dim3(stream_threads()),
                                  args, (size_t)smem, s);
  if (e == cudaErrorCooperativeLaunchTooLarge) {
    (void)cudaGetLastError();
    return BKMOO_OK;
  }
  if (e != cudaSuccess) return BKMOO_ERR_CUDA;
  *taken = true;
  return BKMOO_OK;
}

// Whether a bucket's solve is short enough for the streamed launch, whose
// solver warps are few and on which everything waits.  Frank-Wolfe is one lane's
// fp64 steps, up to max_iter of them (K = 4: 0.9 us a step for MGDA, 2 for
// CAGrad; K = 8: 5 and 13).  Without POLISH every bucket of K >= 3 runs it: 32
// buckets of 25 MiB bf16, K = 4, 256 steps, streamed 4.3 ms (CAGrad 7.9), three
// launches, which solve all buckets at once, 1.3 (1.5).  (K = 2 is exact after
// one line search: 434 us streamed, 639 three.)  With POLISH only buckets whose
// exact solution is not certified do; 1024 steps are 13 ms, far from the 2 s
// after which a wait gives up.
constexpr int32_t kStreamMaxIter = 1024;
bool solve_is_short(int32_t K, int32_t rule, const bkmoo_params& p) {
  if (K == 1 || rule == BKMOO_PCGRAD || rule == BKMOO_MEAN) return true;
  if (K == 2 && rule == BKMOO_MGDA && (p.flags & BKMOO_FLAG_CLOSED_FORM_K2)) return true;
  return p.max_iter <= kStreamMaxIter && (K == 2 || (p.flags & BKMOO_FLAG_POLISH));
}

// Whether a resolve of the view's window takes the streamed launch: the one
// rule behind bkmoo_resolve, bkmoo_resolve_buckets and bkmoo_resolve_launches.
bool streams(const PlanView& v, int32_t rule, const bkmoo_params& p, uint32_t flags) {
  if ((flags & BKMOO_FLAG_THREE_PASS) || !solve_is_short(v.K, rule, p)) return false;
  if (flags & BKMOO_FLAG_FUSED) return v.K <= kStreamMaxK && v.c_hi > v.c_lo;
  return stream_wins(v);
}

// bkmoo_resolve_path's answer (see bkmoo.h); decides nothing.
int choose_path(int32_t K, int32_t dt, int32_t rule, const int64_t* off, int64_t B,
                uint32_t flags) {
  if (flags & BKMOO_FLAG_THREE_PASS) return 0;
  if (flags & BKMOO_FLAG_FUSED) {
    if (K <= 4 && !(flags & BKMOO_FLAG_TEST_WITHHOLD)) return 1;
    return K <= kStreamMaxK ? 2 : 0;
  }
  if (B < 1) return 0;
  if (K <= 2 && B <= 8 && off[B] <= ((int64_t)1 << 22)) return 1;
  if (K < 2 || K > 4) return 0;
  int64_t smax = 0;
  for (int64_t b = 0; b < B; ++b) smax = off[b + 1] - off[b] > smax ? off[b + 1] - off[b] : smax;
  const double mib = 1024.0 * 1024.0;
  const double bytes = (double)smax * elem_bytes(dt), total = bytes * K;
  if (bytes < 2.0 * mib) return 0;
  if (total > 12.0 * mib || (dt != BKMOO_F32 && total < 6.0 * mib)) return 0;
  if (rule == BKMOO_CAGRAD && (dt != BKMOO_F32 || total < 8.0 * mib)) return 0;
  int64_t big = 0;
  for (int64_t b = 0; b < B; ++b)
    if (2 * (off[b + 1] - off[b]) >= smax) big += off[b + 1] - off[b];
  return big * 10 >= off[B] * 9 ? 1 : 0;
}

// The part of a plan view that K, the dtype and the offsets give, as a window
// over the whole plan.
void plan_sizes(int32_t K, int32_t dt, const int64_t* offsets, int64_t B, PlanView* v) {
  const int64_t ch = chunk_elems(dt);
  v->K = K;
  v->in_dtype = dt;
  v->n_buckets = B;
  v->n_chunks = count_chunks(offsets, B, ch);
  v->chunk_elems = ch;
  v->elems = offsets[B];
  v->max_chunks = 0;
  for (int64_t b = 0; b < B; ++b) {
    const int64_t n = (offsets[b + 1] - offsets[b] + ch - 1) / ch;
    if (n > v->max_chunks) v->max_chunks = n;
  }
  full_window(*v);
}

// Common checks of bkmoo_gram / bkmoo_resolve; fills the plan view.
int prepare(const void* const* grads, int32_t K, int32_t dt, const int64_t* offsets,
            int64_t B, void* ws, size_t ws_bytes, PlanView* v, GradPtrs* g) {
  if (K < 1 || K > kMaxK || !dtype_ok(dt) || !grads || !ws) return BKMOO_ERR_INVALID;
  if (!offsets_ok(offsets, B)) return BKMOO_ERR_INVALID;
  if (!aligned(ws, 256)) return BKMOO_ERR_INVALID;
  for (int k = 0; k < K; ++k)
    if (!grads[k] || !aligned(grads[k], 16)) return BKMOO_ERR_INVALID;
  plan_sizes(K, dt, offsets, B, v);
  const WsLayout L = ws_layout(K, B, v->n_chunks);
  if (ws_bytes < L.total_all) return BKMOO_ERR_WORKSPACE;
  char* base = static_cast<char*>(ws);
  v->hdr = reinterpret_cast<WsHeader*>(base);
  v->offsets = reinterpret_cast<const int64_t*>(base + L.offsets);
  v->chunk_prefix = reinterpret_cast<const int64_t*>(base + L.chunk_prefix);
  v->partials = reinterpret_cast<double*>(base + L.partials);
  v->beta = reinterpret_cast<float*>(base + L.beta);
  v->plan_hash = plan_hash(K, dt, offsets, B);
  std::memset(g, 0, sizeof(*g));
  for (int k = 0; k < K; ++k) g->p[k] = grads[k];
  return BKMOO_OK;
}

// Gram pass over the view's window; `reset` clears the workspace status word
// first (once per call of the C ABI, not per window).
// `behind`: the kernels after this pass are launched behind it (not where an
// event is recorded between them).
int launch_gram_pass(const GradPtrs& g, const PlanView& v, cudaStream_t s, bool reset,
                     bool behind) {
  if (reset && cudaMemsetAsync(&v.hdr->status, 0, sizeof(int32_t), s) != cudaSuccess)
    return BKMOO_ERR_CUDA;
  const int64_t nch = v.c_hi - v.c_lo;
  if (nch <= 0) return BKMOO_OK;
  // large K: the variant that prefetches into shared memory (gram_prefetch.cu)
  const bool pf = v.K >= gram_prefetch_min_k();
  const void* fn = pf ? gram_prefetch_fn(v.K, v.in_dtype) : gram_fn(v.K, v.in_dtype);
  int smem = pf ? gram_prefetch_smem(v.K) : 0, threads = kThreads, grid = 0;
  // Fed by bulk copies: with at most a chunk per SM, where a register kernel's
  // CTA has too little in flight alone (64 chunks, K = 2..8: 1.04-1.3 times as
  // fast), and for K = 6 and 7, whose register kernels lose occupancy (3.2 GB: K =
  // 6 bf16 512 -> 464 us, K = 7 fp32 481 -> 448; K = 2..5 and 8 within 3 % either
  // way).  Not for one or two chunks, which gain nothing from the ring but wait
  // for it to be set up (three launches, register / bulk: K = 8 fp32 one chunk
  // 29.0 / 31.2 us, K = 6 bf16 two 25.4 / 27.2, three 30.3 / 29.2).
  int sms = 0;
  if (sm_count(&sms) != cudaSuccess) return BKMOO_ERR_CUDA;
  const void* bulk = gram_bulk_fn(v.K, v.in_dtype);
  if (bulk && nch > 2 && (nch <= sms || v.K == 6 || v.K == 7)) {
    fn = bulk;
    smem = gram_bulk_smem(v.K);
    threads = gram_bulk_threads();
  }
  if (persistent_grid(fn, threads, &grid, smem) != cudaSuccess) return BKMOO_ERR_CUDA;
  if (grid > nch) grid = (int)nch;
  GradPtrs ga = g;
  PlanView va = v;
  void* args[] = {&ga, &va};
  if (cudaLaunchKernel(fn, dim3(grid), dim3(threads), args, smem, s) != cudaSuccess)
    return BKMOO_ERR_CUDA;
  if (launch_group_reduce(v, s, behind) != cudaSuccess) return BKMOO_ERR_CUDA;
  return BKMOO_OK;
}

// The most gradient bytes of a short window, which is combined last chunk first
// (combine_impl.cuh), out of L2, of which a Gram pass just over leaves 50-60 MB; 0
// where the prefetching kernel always is the faster one.  Three launches on
// inputs not in L2 before, the prefetching kernel / this one (us).  Few gradients:
// K = 2 fp32, 40 MB of gradients 39.6 / 36.6, 80 MB 56.0 / 54.8, 120 MB 74.9 / 74.4,
// 390 MB 163.7 / 169.6; K = 3 bf16, 60 MB 47.3 / 44.7, 180 MB 92.7 / 92.3, fp32 290
// MB 118.2 / 123.0; K = 4 fp32, 60 MB 45.6 / 42.6, 105 MB 60.4 / 60.3, 240 MB 115.9
// / 113.9, 390 MB 147.4 / 148.6.  With more to a vector its loads in flight do not
// keep up: K = 4 bf16, 40 MB 41.2 / 43.8, 80 MB 51.4 / 55.8; K = 5 bf16, 63 MB 46.9 /
// 57.6; K = 8 fp32, 80 MB 54.9 / 66.8; K = 16 fp32, 160 MB 110 / 129; K = 11 bf16 and
// K = 12 to 15 fp32 within 4 % either way.  Many bf16 gradients, for which the
// other's slots leave one CTA to an SM: 1.04-1.10 times as fast from 120 to 400 MB,
// 1.02-1.05 to 600, 1.02 at 840, 0.99 at 1200 (K = 16, 160 MB 138 / 127, 420 MB 225
// / 217).  Fewer chunks than SMs: within 2 us either way, at K = 12 to 15 up to 8 %
// slower.  Chunks little more than half full on average at most, every K, as far
// as measured: 1024 buckets of a sixteenth, an eighth and a half of a chunk K = 5 fp32
// 1.14, 1.15 and 1.08 times as fast, K = 8 fp32 1.18, 1.19, 1.02, K = 16 bf16 1.07,
// 1.08, 1.06; 3000 of an eighth and a half K = 4 bf16 1.18, 1.02, K = 7 bf16 1.23,
// 0.97, K = 12 fp32 (1.2 GB) 1.25, 1.02; 1024 of one chunk and 3 elements K = 3 fp32
// 1.12; of whole ones 0.95-1.03.
double last_first_bytes(int K, int dt, bool short_chunks) {
  const double mib = 1024.0 * 1024.0;
  if (short_chunks) return 1024.0 * mib;
  if (K <= (dt == BKMOO_F32 ? 4 : 3)) return 192.0 * mib;
  return dt == BKMOO_BF16 && K >= 12 ? 768.0 * mib : 0.0;
}

int launch_combine(const GradPtrs& g, const PlanView& v, void* out, int32_t out_dtype,
                   cudaStream_t s) {
  const int64_t nch = v.c_hi - v.c_lo;
  if (nch <= 0) return BKMOO_OK;
  const double bytes = (double)v.elems * v.K * elem_bytes(v.in_dtype);
  int sms = 0;
  if (sm_count(&sms) != cudaSuccess) return BKMOO_ERR_CUDA;
  const bool shortw = nch > sms && bytes <= last_first_bytes(v.K, v.in_dtype,
                                                             16 * v.elems <= 9 * nch * v.chunk_elems);
  const void* fn = shortw ? combine_fn(v.K, v.in_dtype, out_dtype)
                          : combine_prefetch_fn(v.K, v.in_dtype, out_dtype);
  const int smem = shortw ? 0 : combine_prefetch_smem(v.K);
  int grid = 0;
  if (persistent_grid(fn, kThreads, &grid, smem) != cudaSuccess) return BKMOO_ERR_CUDA;
  if (grid > nch) grid = (int)nch;
  PlanView va = v;
  GradPtrs ga = g;
  void* outp = out;
  void* args[] = {&ga, &va, &outp};
  if (cudaLaunchKernel(fn, dim3(grid), dim3(kThreads), args, smem, s) != cudaSuccess)
    return BKMOO_ERR_CUDA;
  return BKMOO_OK;
}

bool params_ok(const bkmoo_params& p) {
  return p.max_iter >= 0 && p.cagrad_c >= 0.0 && p.cagrad_c < 1.0 && p.tol >= 0.0;
}

// `flags`: those of prm that count for the call; the withholding test flags only
// with BKMOO_FLAG_FUSED.
SolveParams solve_params(int32_t rule, const bkmoo_params& prm, uint32_t flags) {
  SolveParams sp;
  if (!(flags & BKMOO_FLAG_FUSED))
    flags &= ~(BKMOO_FLAG_TEST_WITHHOLD | BKMOO_FLAG_TEST_WITHHOLD_EXCHANGE);
  sp.rule = rule;
  sp.max_iter = prm.max_iter;
  sp.tol = prm.tol;
  sp.cagrad_c = prm.cagrad_c;
  sp.seed = prm.seed;
  sp.step = prm.step;
  sp.flags = flags;
  return sp;
}

// Checks shared by bkmoo_resolve and bkmoo_resolve_buckets; fills the
// effective parameters, the plan view and the gradient pointers.
int resolve_args(const void* const* grads, int32_t K, int32_t in_dtype, const int64_t* offsets,
                 int64_t n_buckets, int32_t rule, const bkmoo_params* p, const void* out_dir,
                 int32_t out_dtype, void* ws, size_t ws_bytes, bkmoo_params* prm, PlanView* v,
                 GradPtrs* g) {
  if (rule < BKMOO_MGDA || rule > BKMOO_MEAN || !dtype_ok(out_dtype)) return BKMOO_ERR_INVALID;
  if (!out_dir || !aligned(out_dir, 16)) return BKMOO_ERR_INVALID;
  if (p) *prm = *p;
  else bkmoo_default_params(prm);
  if (!params_ok(*prm)) return BKMOO_ERR_INVALID;
  int r = prepare(grads, K, in_dtype, offsets, n_buckets, ws, ws_bytes, v, g);
  if (r != BKMOO_OK) return r;
  // out_dir may be exactly one gradient (same dtype); any other overlap is refused.
  const uintptr_t N = (uintptr_t)offsets[n_buckets];
  const uintptr_t o0 = (uintptr_t)out_dir, o1 = o0 + N * elem_bytes(out_dtype);
  for (int k = 0; k < K; ++k) {
    const uintptr_t g0 = (uintptr_t)grads[k], g1 = g0 + N * elem_bytes(in_dtype);
    if (o0 < g1 && g0 < o1 && !(o0 == g0 && out_dtype == in_dtype)) return BKMOO_ERR_INVALID;
  }
  return BKMOO_OK;
}

// ---------------------------------------------------------------------------
// Host-memory path (bkmoo_resolve_host): windows of whole buckets streamed
// through three device staging slots (measured on GB300: 3-5 % faster end to
// end than two, whose output copies held back the next windows' inputs).
// ---------------------------------------------------------------------------

constexpr int kHostSlots = 3;

// Each slot has K input regions and one output region, each 256-byte
// aligned, with one 16-byte vector of slack so that a window may start at
// any element and still keep vector alignment.
size_t region_bytes(int64_t elems, int32_t dt) {
  return align256((size_t)elems * elem_bytes(dt) + 16);
}

size_t staging_bytes_for(int32_t K, int32_t dti, int32_t dto, int64_t elems) {
  return (size_t)kHostSlots * ((size_t)K * region_bytes(elems, dti) + region_bytes(elems, dto));
}

// Elements of one language a slot holds for a staging buffer of `bytes`: the
// largest cap with staging_bytes_for(cap) <= bytes.
int64_t slot_capacity(int32_t K, int32_t dti, int32_t dto, size_t bytes) {
  const int64_t per_elem = K * elem_bytes(dti) + elem_bytes(dto);
  int64_t lo = 0, hi = (int64_t)(bytes / kHostSlots) / per_elem + 1;  // fits, does not fit
  if (staging_bytes_for(K, dti, dto, 0) > bytes) return 0;
  while (hi - lo > 1) {
    const int64_t mid = lo + (hi - lo) / 2;
    if (staging_bytes_for(K, dti, dto, mid) <= bytes) lo = mid;
    else hi = mid;
  }
  return lo;
}

}  // namespace

cudaError_t bkmoo::sm_count(int* n) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  LaunchCache& c = cache();
  std::lock_guard<std::mutex> lk(c.mu);
  return device_sms(c, dev, n);
}

extern "C" {

void bkmoo_default_params(bkmoo_params* p) {
  if (!p) return;
  p->max_iter = 256;
  p->tol = 1e-12;
  p->cagrad_c = 0.5;
  p->seed = 0;
  p->step = 0;
  p->flags = BKMOO_FLAG_CLOSED_FORM_K2 | BKMOO_FLAG_POLISH;
  p->events = nullptr;
}

int bkmoo_plan(const int64_t* param_sizes, int32_t n_params, int32_t elem_bytes_,
               int64_t bucket_bytes, int64_t* out_offsets, int64_t out_cap,
               int64_t* n_buckets) {
  if (!n_buckets || n_params < 0 || (n_params > 0 && !param_sizes) || elem_bytes_ <= 0 ||
      bucket_bytes <= 0)
    return BKMOO_ERR_INVALID;
  const int64_t cap = bucket_bytes / elem_bytes_;
  if (cap < 1) return BKMOO_ERR_INVALID;
  for (int32_t i = 0; i < n_params; ++i)
    if (param_sizes[i] < 0) return BKMOO_ERR_INVALID;

  // Walk the tensors last-registered first; `fill` is the open bucket's size
  // and `end` the flat position reached so far.
  std::vector<int64_t> bounds;
  bounds.push_back(0);
  int64_t fill = 0, end = 0;
  for (int32_t i = n_params; i-- > 0;) {
    int64_t left = param_sizes[i];
    if (left == 0) continue;
    if (fill > 0 && fill + left > cap) {  // does not fit: close the open bucket
      bounds.push_back(end);
      fill = 0;
    }
    while (left > cap) {  // oversize tensor: whole cap-sized pieces
      end += cap;
      bounds.push_back(end);
      left -= cap;
    }
    fill += left;
    end += left;
  }
  if (fill > 0) bounds.push_back(end);
  *n_buckets = (int64_t)bounds.size() - 1;
  if (!out_offsets) return BKMOO_OK;
  if (out_cap < (int64_t)bounds.size()) return BKMOO_ERR_BUFFER_TOO_SMALL;
  std::memcpy(out_offsets, bounds.data(), sizeof(int64_t) * bounds.size());
  return BKMOO_OK;
}

int bkmoo_workspace_size(int32_t K, int32_t in_dtype, const int64_t* offsets,
                         int64_t n_buckets, size_t* bytes) {
  if (!bytes || K < 1 || K > kMaxK || !dtype_ok(in_dtype) || !offsets_ok(offsets, n_buckets))
    return BKMOO_ERR_INVALID;
  const int64_t nch = count_chunks(offsets, n_buckets, chunk_elems(in_dtype));
  *bytes = ws_layout(K, n_buckets, nch).total_all;
  return BKMOO_OK;
}

int bkmoo_workspace_init(int32_t K, int32_t in_dtype, const int64_t* offsets,
                         int64_t n_buckets, void* ws, size_t ws_bytes, void* stream) {
  if (K < 1 || K > kMaxK || !dtype_ok(in_dtype) || !ws || !aligned(ws, 256) ||
      !offsets_ok(offsets, n_buckets))
    return BKMOO_ERR_INVALID;
  const int64_t ch = chunk_elems(in_dtype);
  const int64_t nch = count_chunks(offsets, n_buckets, ch);
  const WsLayout L = ws_layout(K, n_buckets, nch);
  if (ws_bytes < L.total_all) return BKMOO_ERR_WORKSPACE;
  // Host image of header + bucket table, copied in one transfer.
  std::vector<unsigned char> img(L.partials, 0);
  WsHeader h;
  std::memset(&h, 0, sizeof h);
  h.magic = kMagic;
  h.K = K;
  h.in_dtype = in_dtype;
  h.status = BKMOO_OK;
  h.n_buckets = n_buckets;
  h.n_elems = offsets[n_buckets];
  h.n_chunks = nch;
  h.chunk_elems = ch;
  h.plan_hash = plan_hash(K, in_dtype, offsets, n_buckets);
  std::memcpy(img.data(), &h, sizeof h);
  std::memcpy(img.data() + L.offsets, offsets, sizeof(int64_t) * (size_t)(n_buckets + 1));
  int64_t* cp = reinterpret_cast<int64_t*>(img.data() + L.chunk_prefix);
  cp[0] = 0;
  for (int64_t b = 0; b < n_buckets; ++b) cp[b + 1] = cp[b] + (offsets[b + 1] - offsets[b] + ch - 1) / ch;
  // The bucket of every chunk (streamed path).
  std::vector<int32_t> cb((size_t)nch);
  for (int64_t b = 0; b < n_buckets; ++b)
    for (int64_t c = cp[b]; c < cp[b + 1]; ++c) cb[(size_t)c] = (int32_t)b;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemcpyAsync(ws, img.data(), img.size(), cudaMemcpyHostToDevice, s) != cudaSuccess)
    return BKMOO_ERR_CUDA;
  if (nch > 0 && cudaMemcpyAsync(static_cast<char*>(ws) + L.chunk_bucket, cb.data(),
                                 sizeof(int32_t) * (size_t)nch, cudaMemcpyHostToDevice,
                                 s) != cudaSuccess)
    return BKMOO_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return BKMOO_ERR_CUDA;
  return BKMOO_OK;
}

int bkmoo_gram(const void* const* grads, int32_t K, int32_t in_dtype, const int64_t* offsets,
               int64_t n_buckets, double* out_gram, void* ws, size_t ws_bytes, void* stream) {
  if (!out_gram && n_buckets > 0) return BKMOO_ERR_INVALID;
  PlanView v;
  GradPtrs g;
  int r = prepare(grads, K, in_dtype, offsets, n_buckets, ws, ws_bytes, &v, &g);
  if (r != BKMOO_OK) return r;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  r = launch_gram_pass(g, v, s, true, true);
  if (r != BKMOO_OK) return r;
  if (launch_gram_finalize(v, out_gram, s, true) != cudaSuccess) return BKMOO_ERR_CUDA;
  return BKMOO_OK;
}

int bkmoo_resolve(const void* const* grads, int32_t K, int32_t in_dtype, const int64_t* offsets,
                  int64_t n_buckets, int32_t rule, const bkmoo_params* p, void* out_dir,
                  int32_t out_dtype, float* out_weights, int32_t* out_status, void* ws,
                  size_t ws_bytes, void* stream) {
  bkmoo_params prm;
  PlanView v;
  GradPtrs g;
  int r = resolve_args(grads, K, in_dtype, offsets, n_buckets, rule, p, out_dir, out_dtype, ws,
                       ws_bytes, &prm, &v, &g);
  if (r != BKMOO_OK) return r;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaEvent_t* ev = static_cast<cudaEvent_t*>(prm.events);
  const SolveParams sp = solve_params(rule, prm, prm.flags);
  if (ev && cudaEventRecord(ev[0], s) != cudaSuccess) return BKMOO_ERR_CUDA;
  if (streams(v, rule, prm, prm.flags)) {
    bool taken = false;
    r = launch_stream(g, v, sp, ws, out_weights, out_status, out_dir, out_dtype, true, &taken, s);
    if (r != BKMOO_OK) return r;
    if (taken) {
      for (int i = 1; i < 4; ++i)
        if (ev && cudaEventRecord(ev[i], s) != cudaSuccess) return BKMOO_ERR_CUDA;
      return BKMOO_OK;
    }
  }
  r = launch_gram_pass(g, v, s, true, !ev);
  if (r != BKMOO_OK) return r;
  if (ev && cudaEventRecord(ev[1], s) != cudaSuccess) return BKMOO_ERR_CUDA;
  if (launch_solve(v, sp, out_weights, out_status, s, !ev) != cudaSuccess) return BKMOO_ERR_CUDA;
  if (ev && cudaEventRecord(ev[2], s) != cudaSuccess) return BKMOO_ERR_CUDA;
  r = launch_combine(g, v, out_dir, out_dtype, s);
  if (r != BKMOO_OK) return r;
  if (ev && cudaEventRecord(ev[3], s) != cudaSuccess) return BKMOO_ERR_CUDA;
  return BKMOO_OK;
}

int bkmoo_resolve_buckets(const void* const* grads, int32_t K, int32_t in_dtype,
                          const int64_t* offsets, int64_t n_buckets, int64_t b_lo, int64_t b_hi,
                          int32_t rule, const bkmoo_params* p, void* out_dir, int32_t out_dtype,
                          float* out_weights, int32_t* out_status, void* ws, size_t ws_bytes,
                          void* stream) {
  bkmoo_params prm;
  PlanView v;
  GradPtrs g;
  int r = resolve_args(grads, K, in_dtype, offsets, n_buckets, rule, p, out_dir, out_dtype, ws,
                       ws_bytes, &prm, &v, &g);
  if (r != BKMOO_OK) return r;
  if (b_lo < 0 || b_hi > n_buckets || b_lo > b_hi) return BKMOO_ERR_INVALID;
  if (b_lo == b_hi) return BKMOO_OK;
  v.b_lo = b_lo;
  v.b_hi = b_hi;
  int64_t c = 0;
  for (int64_t b = 0; b < b_lo; ++b) c += (offsets[b + 1] - offsets[b] + v.chunk_elems - 1) / v.chunk_elems;
  v.c_lo = c;
  for (int64_t b = b_lo; b < b_hi; ++b) c += (offsets[b + 1] - offsets[b] + v.chunk_elems - 1) / v.chunk_elems;
  v.c_hi = c;
  v.elems = offsets[b_hi] - offsets[b_lo];
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint32_t flags = prm.flags & ~BKMOO_FLAG_FUSED;
  const SolveParams sp = solve_params(rule, prm, flags);
  // One or two buckets: the three launches, which share the SMs with whatever
  // the caller overlaps them with; the streamed launch needs all of them at
  // once (a training step that resolves each bucket beside the backward pass:
  // 263.9 ms with three launches per bucket, 267.3 streamed).
  if (b_hi - b_lo > 2 && streams(v, rule, prm, flags)) {
    bool taken = false;
    r = launch_stream(g, v, sp, ws, out_weights, out_status, out_dir, out_dtype, false, &taken, s);
    if (r != BKMOO_OK || taken) return r;
  }
  r = launch_gram_pass(g, v, s, false, true);
  if (r != BKMOO_OK) return r;
  if (launch_solve(v, sp, out_weights, out_status, s, true) != cudaSuccess) return BKMOO_ERR_CUDA;
  return launch_combine(g, v, out_dir, out_dtype, s);
}

int bkmoo_host_staging_size(int32_t K, int32_t in_dtype, int32_t out_dtype,
                            const int64_t* offsets, int64_t n_buckets, int64_t window_elems,
                            size_t* bytes) {
  if (!bytes || K < 1 || K > kMaxK || !dtype_ok(in_dtype) || !dtype_ok(out_dtype) ||
      !offsets_ok(offsets, n_buckets) || window_elems < 0)
    return BKMOO_ERR_INVALID;
  int64_t w = window_elems;
  for (int64_t b = 0; b < n_buckets; ++b)
    if (offsets[b + 1] - offsets[b] > w) w = offsets[b + 1] - offsets[b];
  *bytes = staging_bytes_for(K, in_dtype, out_dtype, w);
  return BKMOO_OK;
}

int bkmoo_resolve_host(const void* const* host_grads, int32_t K, int32_t in_dtype,
                       const int64_t* offsets, int64_t n_buckets, int32_t rule,
                       const bkmoo_params* p, void* host_out, int32_t out_dtype,
                       float* out_weights, int32_t* out_status, void* ws, size_t ws_bytes,
                       void* staging, size_t staging_bytes, void* stream) {
  if (rule < BKMOO_MGDA || rule > BKMOO_MEAN || !dtype_ok(out_dtype) || !host_out || !staging ||
      !aligned(staging, 256))
    return BKMOO_ERR_INVALID;
  bkmoo_params prm;
  if (p) prm = *p;
  else bkmoo_default_params(&prm);
  if (!params_ok(prm)) return BKMOO_ERR_INVALID;
  // The kernels address the staging slots, never the host buffers; `prepare`
  // checks the plan and workspace (its pointer checks see the host pointers).
  PlanView v;
  GradPtrs unused;
  int r = prepare(host_grads, K, in_dtype, offsets, n_buckets, ws, ws_bytes, &v, &unused);
  if (r != BKMOO_OK) return r;
  const int ei = elem_bytes(in_dtype), eo = elem_bytes(out_dtype);
  const int64_t N = offsets[n_buckets];
  {  // host_out may be exactly one gradient (same dtype); any other overlap is refused.
    const uintptr_t o0 = (uintptr_t)host_out, o1 = o0 + (uintptr_t)N * eo;
    for (int k = 0; k < K; ++k) {
      const uintptr_t g0 = (uintptr_t)host_grads[k], g1 = g0 + (uintptr_t)N * ei;
      if (o0 < g1 && g0 < o1 && !(o0 == g0 && out_dtype == in_dtype)) return BKMOO_ERR_INVALID;
    }
  }
  const int64_t cap = slot_capacity(K, in_dtype, out_dtype, staging_bytes);
  for (int64_t b = 0; b < n_buckets; ++b)
    if (offsets[b + 1] - offsets[b] > cap) return BKMOO_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(&v.hdr->status, 0, sizeof(int32_t), s) != cudaSuccess)
    return BKMOO_ERR_CUDA;
  if (n_buckets == 0) return BKMOO_OK;
  const SolveParams sp = solve_params(rule, prm, prm.flags);

  // Slot layout: K input regions then the output region, each of
  // region_bytes(cap) bytes.
  const size_t rin = region_bytes(cap, in_dtype), rout = region_bytes(cap, out_dtype);
  const size_t slot_bytes = (size_t)K * rin + rout;
  char* const stage = static_cast<char*>(staging);
  const int vec_in = 16 / ei;  // elements per 16-byte input vector

  // Copy streams and events live for this call only; destroying them while
  // work is queued is legal (their resources go once the work completes).
  cudaStream_t h2d = nullptr, d2h = nullptr;
  cudaEvent_t ev_start = nullptr, in_ready[kHostSlots] = {}, in_free[kHostSlots] = {},
              out_ready[kHostSlots] = {}, out_free[kHostSlots] = {};
  bool ok = cudaStreamCreateWithFlags(&h2d, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamCreateWithFlags(&d2h, cudaStreamNonBlocking) == cudaSuccess &&
            cudaEventCreateWithFlags(&ev_start, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; ok && i < kHostSlots; ++i)
    ok = cudaEventCreateWithFlags(&in_ready[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&in_free[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&out_ready[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&out_free[i], cudaEventDisableTiming) == cudaSuccess;
  // Both copy streams start after the work already queued on `stream`.
  ok = ok && cudaEventRecord(ev_start, s) == cudaSuccess &&
       cudaStreamWaitEvent(h2d, ev_start, 0) == cudaSuccess &&
       cudaStreamWaitEvent(d2h, ev_start, 0) == cudaSuccess;

  const int64_t ch = v.chunk_elems;
  int64_t b0 = 0, c_next = 0;
  for (int64_t win = 0; ok && b0 < n_buckets; ++win) {
    // the window: whole buckets b0 .. b1-1, at most `cap` elements
    int64_t b1 = b0 + 1;
    while (b1 < n_buckets && offsets[b1 + 1] - offsets[b0] <= cap) ++b1;
    const int slot = (int)(win % kHostSlots);
    const int64_t lo = offsets[b0], hi = offsets[b1], n = hi - lo;
    // element `lo` sits at the same offset within a 16-byte vector as in a
    // 16-byte-aligned buffer, so the kernels' vector/scalar split holds
    const int64_t base = lo / vec_in * vec_in;
    char* sin = stage + (size_t)slot * slot_bytes;
    char* sout = sin + (size_t)K * rin;
    if (win >= kHostSlots) ok = ok && cudaStreamWaitEvent(h2d, in_free[slot], 0) == cudaSuccess;
    for (int k = 0; ok && k < K; ++k)
      ok = cudaMemcpyAsync(sin + (size_t)k * rin + (size_t)(lo - base) * ei,
                           static_cast<const char*>(host_grads[k]) + (size_t)lo * ei,
                           (size_t)n * ei, cudaMemcpyHostToDevice, h2d) == cudaSuccess;
    ok = ok && cudaEventRecord(in_ready[slot], h2d) == cudaSuccess;

    // Kernel pointers are shifted so that global element i of the plan is
    // addressed at (region + (i - base) * e): only [lo, hi) is touched.
    GradPtrs gw;
    std::memset(&gw, 0, sizeof gw);
    for (int k = 0; k < K; ++k)
      gw.p[k] = reinterpret_cast<const void*>((uintptr_t)(sin + (size_t)k * rin) -
                                              (uintptr_t)base * ei);
    void* outw = reinterpret_cast<void*>((uintptr_t)sout - (uintptr_t)base * eo);
    PlanView vw = v;
    vw.b_lo = b0;
    vw.b_hi = b1;
    vw.elems = n;
    // chunk range of the window: chunks are numbered bucket by bucket
    vw.c_lo = c_next;
    for (int64_t b = b0; b < b1; ++b) c_next += (offsets[b + 1] - offsets[b] + ch - 1) / ch;
    vw.c_hi = c_next;
    ok = ok && cudaStreamWaitEvent(s, in_ready[slot], 0) == cudaSuccess;
    if (win >= kHostSlots) ok = ok && cudaStreamWaitEvent(s, out_free[slot], 0) == cudaSuccess;
    if (ok) r = launch_gram_pass(gw, vw, s, false, true);
    ok = ok && r == BKMOO_OK &&
         launch_solve(vw, sp, out_weights, out_status, s, true) == cudaSuccess;
    if (ok) r = launch_combine(gw, vw, outw, out_dtype, s);
    ok = ok && r == BKMOO_OK && cudaEventRecord(in_free[slot], s) == cudaSuccess &&
         cudaEventRecord(out_ready[slot], s) == cudaSuccess;

    ok = ok && cudaStreamWaitEvent(d2h, out_ready[slot], 0) == cudaSuccess &&
         cudaMemcpyAsync(static_cast<char*>(host_out) + (size_t)lo * eo,
                         sout + (size_t)(lo - base) * eo, (size_t)n * eo,
                         cudaMemcpyDeviceToHost, d2h) == cudaSuccess &&
         cudaEventRecord(out_free[slot], d2h) == cudaSuccess;
    b0 = b1;
  }
  // `stream` completes only after the last copy back.
  ok = ok && cudaEventRecord(ev_start, d2h) == cudaSuccess &&
       cudaStreamWaitEvent(s, ev_start, 0) == cudaSuccess;
  if (h2d) cudaStreamDestroy(h2d);
  if (d2h) cudaStreamDestroy(d2h);
  if (ev_start) cudaEventDestroy(ev_start);
  for (int i = 0; i < kHostSlots; ++i) {
    if (in_ready[i]) cudaEventDestroy(in_ready[i]);
    if (in_free[i]) cudaEventDestroy(in_free[i]);
    if (out_ready[i]) cudaEventDestroy(out_ready[i]);
    if (out_free[i]) cudaEventDestroy(out_free[i]);
  }
  if (!ok) return r != BKMOO_OK ? r : BKMOO_ERR_CUDA;
  return BKMOO_OK;
}

int bkmoo_workspace_status(const void* ws, void* stream, int32_t* status) {
  if (!ws || !status || !aligned(ws, 256)) return BKMOO_ERR_INVALID;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaStreamSynchronize(s) != cudaSuccess) return BKMOO_ERR_CUDA;
  const WsHeader* h = static_cast<const WsHeader*>(ws);
  int32_t st = 0;
  if (cudaMemcpy(&st, &h->status, sizeof st, cudaMemcpyDeviceToHost) != cudaSuccess)
    return BKMOO_ERR_CUDA;
  *status = st;
  return BKMOO_OK;
}

const char* bkmoo_status_string(int32_t status) {
  switch (status) {
    case BKMOO_OK: return "ok";
    case BKMOO_ERR_INVALID: return "invalid argument";
    case BKMOO_ERR_CUDA: return "CUDA error";
    case BKMOO_ERR_NONFINITE: return "non-finite Gram matrix (beta = 1/K)";
    case BKMOO_ERR_WORKSPACE: return "workspace too small or not initialised for this plan";
    case BKMOO_ERR_TIMEOUT: return "bounded device wait timed out";
    case BKMOO_ERR_BUFFER_TOO_SMALL: return "output buffer too small";
    case BKMOO_ERR_NOT_CONVERGED: return "solver stopped at its iteration cap";
    default: return "unknown status";
  }
}

int32_t bkmoo_version(void) { return kVersion; }

int bkmoo_resolve_path(int32_t K, int32_t in_dtype, int32_t rule, const int64_t* offsets,
                       int64_t n_buckets, uint32_t flags, int32_t* path) {
  if (!path || K < 1 || K > kMaxK || !dtype_ok(in_dtype) || rule < BKMOO_MGDA ||
      rule > BKMOO_MEAN || !offsets_ok(offsets, n_buckets))
    return BKMOO_ERR_INVALID;
  *path = choose_path(K, in_dtype, rule, offsets, n_buckets, flags);
  return BKMOO_OK;
}

int bkmoo_resolve_launches(int32_t K, int32_t in_dtype, int32_t rule, const int64_t* offsets,
                           int64_t n_buckets, const bkmoo_params* p, int32_t* launches) {
  if (!launches || K < 1 || K > kMaxK || !dtype_ok(in_dtype) || rule < BKMOO_MGDA ||
      rule > BKMOO_MEAN || !offsets_ok(offsets, n_buckets))
    return BKMOO_ERR_INVALID;
  bkmoo_params prm;
  if (p) prm = *p;
  else bkmoo_default_params(&prm);
  if (!params_ok(prm)) return BKMOO_ERR_INVALID;
  PlanView v;
  std::memset(&v, 0, sizeof v);
  plan_sizes(K, in_dtype, offsets, n_buckets, &v);
  if (n_buckets == 0) *launches = 0;
  else if (streams(v, rule, prm, prm.flags)) *launches = 1;
  else *launches = v.max_chunks > kGroupMinChunks ? 4 : 3;
  return BKMOO_OK;
}

int bkmoo_selftest_fp64(int32_t op, const double* a, const double* b, double* out, int64_t n,
                        void* stream) {
  if ((op != 0 && op != 1) || n < 0 || (n > 0 && (!a || !out || (op == 0 && !b))))
    return BKMOO_ERR_INVALID;
  return launch_selftest_fp64(op, a, b, out, n, static_cast<cudaStream_t>(stream)) == cudaSuccess
             ? BKMOO_OK
             : BKMOO_ERR_CUDA;
}

}  // extern "C"
