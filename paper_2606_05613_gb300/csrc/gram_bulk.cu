// Gram pass fed by bulk copies: one producer warp keeps a ring of stages (one
// or two 16-byte vectors of each gradient for each of 256 threads) in flight
// by cp.async.bulk, eight Gram warps take each stage from shared memory.  The
// chunks, thread layout, order of every sum and the partials are those of
// gram_partials_kernel, bit for bit.
//
// What bounds it: HBM reads; on a plan of few chunks, the bytes that one SM
// has in flight.  A register kernel's CTA has two vectors of each gradient
// per thread in flight, in bursts between which it computes, and needs several
// CTAs per SM to fill the gaps; here about 100 KB per CTA are in flight whatever
// the warps do.  K = 4, 64 chunks of fp32: 20.9 -> 16.2 us for the Gram call; K =
// 6 bf16, 3.2 GB: 512 -> 464 us (6.9 TB/s).
#include "bulk_copy.cuh"
#include "gram_prefetch.cuh"

namespace bkmoo {
namespace {

constexpr int kBulkThreads = kThreads + 32;
constexpr uint64_t kBulkWaitNs = 4000000000ull;

constexpr int bulk_items(int K) { return K <= 2 ? 4 : K <= 4 ? 2 : 1; }
constexpr int bulk_stage_bytes(int K) { return K * bulk_items(K) * kThreads * 16; }
// two CTAs per SM
constexpr int bulk_stages(int K) { return 100 * 1024 / bulk_stage_bytes(K); }

struct BulkChunk {
  int64_t s, vs, ve, e;
  int32_t nv;
};

// Bounded wait on a barrier of this CTA, the same answer on every lane.
__device__ __forceinline__ bool bulk_wait(uint64_t* bar, unsigned parity, volatile int* abort,
                                          WsHeader* h) {
  uint64_t t0 = 0;
  for (unsigned it = 0;; ++it) {
    if (__all_sync(0xffffffffu, bar_try(bar, parity))) return true;
    if ((it & 63u) == 63u) {
      const uint64_t t = stream_ns();
      if (t0 == 0) t0 = t;
      const bool late = t - t0 > kBulkWaitNs;
      if (late) {
        *abort = 1;
        record_error(h, BKMOO_ERR_TIMEOUT);
      }
      if (__any_sync(0xffffffffu, late || *abort != 0)) return false;
    }
  }
}

template <int K, int DT>
__global__ void __launch_bounds__(kBulkThreads, 2)
    gram_bulk_kernel(const GradPtrs g, const PlanView v) {
  constexpr int P = tri(K), EPV = elems_per_vec(DT), EB = 16 / EPV;
  constexpr int U = bulk_items(K), SV = U * kThreads, SB = bulk_stage_bytes(K);
  constexpr int N = bulk_stages(K), kDesc = 16;
  static_assert(N <= 12, "descriptors in flight");
  extern __shared__ unsigned char gb_dyn[];
  __shared__ float red[kWarps][P];
  __shared__ uint64_t full[N], empty[N];
  __shared__ BulkChunk desc[kDesc];
  __shared__ volatile int abort;

  grid_release();
  if (!header_ok(v)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) record_error(v.hdr, BKMOO_ERR_WORKSPACE);
    return;
  }
  unsigned char* ring =
      reinterpret_cast<unsigned char*>(((uintptr_t)gb_dyn + 127) & ~(uintptr_t)127);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
  if (t == 0) {
    for (int i = 0; i < N; ++i) {
      bar_init(&full[i], 1);
      bar_init(&empty[i], kWarps);
    }
    abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  int slot = 0, i = 0;
  if (wid == kWarps) {
    // producer: chunk i's geometry is searched while the ring is full
    const uint64_t pol = stream_policy(false);
    BucketTracker bt;
    bt.init(v);
    unsigned par = 1;
    uint32_t issued = 0;
    for (int64_t w = v.c_lo + blockIdx.x; w < v.c_hi; w += gridDim.x, ++i) {
      BulkChunk c;
      bt.seek(v, w);
      c.s = bt.o0 + (w - bt.c0) * v.chunk_elems;
      c.e = min(c.s + v.chunk_elems, bt.o1);
      c.vs = (c.s + EPV - 1) / EPV * EPV;
      if (c.vs > c.e) c.vs = c.e;
      c.ve = c.e / EPV * EPV;
      if (c.ve < c.vs) c.ve = c.vs;
      c.nv = (int)((c.ve - c.vs) / EPV);
      const int n = c.nv > SV ? (c.nv + SV - 1) / SV : 1;
      int64_t off = c.vs * EB;
      bool on = true;
      for (int s = 0; s < n && on; ++s, off += SV * 16) {
        on = bulk_wait(&empty[slot], par, &abort, v.hdr);
        if (!on) break;
        if (s == 0) {
          if (lane == 0) desc[i % kDesc] = c;
          __syncwarp();
        }
        const int left = c.nv - s * SV;
        const unsigned bytes = left > 0 ? (unsigned)(left < SV ? left : SV) * 16u : 0u;
        if (elect_one()) {
          bar_arrive_tx(&full[slot], bytes * K);
          if (bytes) {
#pragma unroll
            for (int k = 0; k < K; ++k)
              bulk_load(ring + slot * SB + k * (SV * 16), static_cast<const char*>(g.p[k]) + off,
                        bytes, &full[slot], pol);
          }
        }
        ++issued;
        if (++slot == N) {
          slot = 0;
          par ^= 1;
        }
      }
      if (!on) break;
    }
    // every copy has landed before the CTA may end
    for (int k = 0; k < N && (uint32_t)k < issued; ++k) {
      const unsigned last = ((issued - 1 - k) / N) & 1u;
      for (unsigned it = 0; it < 4000000u && !bar_try(&full[k], last); ++it) {
      }
    }
    return;
  }
  unsigned par = 0;
  for (int64_t w = v.c_lo + blockIdx.x; w < v.c_hi; w += gridDim.x, ++i) {
    float acc[P];
#pragma unroll
    for (int p = 0; p < P; ++p) acc[p] = 0.0f;
    int n = 1, nv = 0, nh = 0, nt = 0;
    float xs[K];
    for (int s = 0; s < n; ++s) {
      // (once it gives up it gives up on every warp, which then only keep
      // the CTA's barriers in step)
      if (!bulk_wait(&full[slot], par, &abort, v.hdr)) break;
      if (s == 0) {
        const BulkChunk& c = desc[i % kDesc];
        nv = c.nv;
        n = nv > SV ? (nv + SV - 1) / SV : 1;
        nh = (int)(c.vs - c.s);
        nt = (int)(c.e - c.ve);
        if (t < nh + nt) {
          const int64_t sc = t < nh ? c.s + t : c.ve + (t - nh);
#pragma unroll
          for (int k = 0; k < K; ++k) xs[k] = load_scalar<DT>(g.p[k], sc);
        }
      }
      const unsigned char* sb = ring + slot * SB + t * 16;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        uint4 r[K];
#pragma unroll
        for (int k = 0; k < K; ++k)
          r[k] = *reinterpret_cast<const uint4*>(sb + (k * U + u) * (kThreads * 16));
        if (u == U - 1) {
          __syncwarp();
          if (lane == 0) bar_arrive(&empty[slot]);
        }
        if ((s * U + u) * kThreads + t < nv) gram_accumulate<K, DT>(acc, r);
      }
      if (++slot == N) {
        slot = 0;
        par ^= 1;
      }
    }
    if (t < nh + nt) {
      int p = 0;
#pragma unroll
      for (int a = 0; a < K; ++a)
#pragma unroll
        for (int b = a; b < K; ++b) {
          acc[p] = fmaf(xs[a], xs[b], acc[p]);
          ++p;
        }
    }
    // the chunk's partials, as cta_reduce_store forms them (the producer warp
    // takes no part in the barrier)
    __syncwarp();
#pragma unroll
    for (int p = 0; p < P; ++p) {
      float x = acc[p];
      x += __shfl_down_sync(0xffffffffu, x, 16);
      x += __shfl_down_sync(0xffffffffu, x, 8);
      x += __shfl_down_sync(0xffffffffu, x, 4);
      x += __shfl_down_sync(0xffffffffu, x, 2);
      x += __shfl_down_sync(0xffffffffu, x, 1);
      if (lane == 0) red[wid][p] = x;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
    for (int p = t; p < P; p += kThreads) {
      double x = 0.0;
#pragma unroll
      for (int q = 0; q < kWarps; ++q) x += (double)red[q][p];
      v.partials[w * P + p] = x;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
  }
}

#define BKMOO_BULK_TABLE(DT)                                                              \
  {(const void*)gram_bulk_kernel<2, DT>, (const void*)gram_bulk_kernel<3, DT>,              \
   (const void*)gram_bulk_kernel<4, DT>, (const void*)gram_bulk_kernel<5, DT>,              \
   (const void*)gram_bulk_kernel<6, DT>, (const void*)gram_bulk_kernel<7, DT>,              \
   (const void*)gram_bulk_kernel<8, DT>}
static const void* const kBulkF32[kBulkMaxK - kBulkMinK + 1] = BKMOO_BULK_TABLE(BKMOO_F32);
static const void* const kBulkBf16[kBulkMaxK - kBulkMinK + 1] = BKMOO_BULK_TABLE(BKMOO_BF16);

}  // namespace

const void* gram_bulk_fn(int K, int dt) {
  if (K < kBulkMinK || K > kBulkMaxK) return nullptr;
  return dt == BKMOO_F32 ? kBulkF32[K - kBulkMinK] : kBulkBf16[K - kBulkMinK];
}
int gram_bulk_smem(int K) { return bulk_stages(K) * bulk_stage_bytes(K) + 128; }
int gram_bulk_threads() { return kBulkThreads; }

}  // namespace bkmoo
