// Streamed resolve: Gram -> solve -> combination of a window of the plan in
// one co-resident launch, one CTA per SM, in which the combination of a bucket
// runs a few microseconds behind its Gram, so that most of what it needs is
// still on the chip (Algorithm 1 resolves each bucket as soon as it is full).
//
// What bounds it: HBM.  The three launches read the gradients twice,
// (2K + 1) e bytes per element with the output; here a chunk's vectors stay in
// tensor memory (256 KB per SM that this path has no matrix product for) or
// are asked to stay in L2 between their two uses, and only the rest is read
// again.  Measured under ncu, GPT-2 small (K = 4 fp32, 25 MiB buckets): 3.36
// GB of DRAM traffic for 1.99 GB of gradients (4.48 with two reads) at 6.6 TB/s;
// 120 M fp32 elements in 1 MiB buckets: 2.67 GB for 1.92 (4.32).  What is kept is
// set by the bytes in flight between the two uses (a bucket, the solve's chain,
// the copy rings) against 39 MB of tensor memory and about 55 MB of L2 (of 126
// MB: a probe that re-reads a stream D bytes later finds all of it up to D = 60
// MB with evict_last, 45 MB of it at D = 120 MB), so a shorter chain means fewer
// bytes.  Three launches against this one (us): GPT-2 small 672, 520; 250 M fp32
// elements K = 4 in 1 MiB buckets 1279, 820; 500 M K = 2 in 4 MiB buckets 1496, 882.
//
// Chunks and arithmetic are those of the three launches: the same chunks, the
// same thread for every vector, the same order of every sum, so the results
// are the same bit for bit.  Chunk w0 + i belongs to CTA i mod n_stream.
//
// A streaming CTA has 16 warps:
//   0-7   Gram: consume the Gram ring, one chunk after the other, leave the
//         stages marked for it in tensor memory.
//   8-11  combination: wait for the bucket's coefficients, then take each
//         stage from tensor memory or from the combination ring.  Warp c reads
//         the tensor-memory lanes that Gram warps c and c + 4 wrote.
//   12    Gram producer: bulk copies into the Gram ring (4-6 stages of 20-32
//         KiB).  Decides per stage, as slots are free at that moment, whether
//         it is kept in tensor memory, asked to stay in L2 (evict_last, a
//         bounded number of bytes) or read again from wherever it is
//         (evict_first).  Never more than `lead` stages ahead of the
//         combination, except within its bucket and the next.
//   13    rows: sums the Gram warps' triangles of a chunk (fp64) and publishes
//         the row.
//   14    combination producer: follows chunk by chunk and copies again the
//         stages that are not in tensor memory, as half stages.
//   15    idle (warps are allocated in fours).
// One elected lane issues the K copies of a stage; with a copy per lane the
// producers, not memory, set the pace (qwen-shaped plan: 765 ns per stage).
//
// The last n_solve CTAs only solve: teams of 2-8 warps sum a bucket's rows as
// they arrive, solve and publish.  On a streaming SM a K = 4 MGDA solve takes
// 10 us instead of 4 to 5, and everything waits for it.
//
// Hand-offs between CTAs are single 64-bit words that are 0 until written
// (cleared by a memset before the launch): no fence, no counter, and the poll
// that finds a word has its value.  No wait closes a cycle: the Gram of a
// bucket waits for no coefficients of it or of a later bucket.  Waits for
// another CTA give up after 2 s: BKMOO_ERR_TIMEOUT in the workspace status
// word, a flag in the window's rows that ends every other wait, and each CTA
// lets its copies land and returns.
#pragma once

#include "bulk_copy.cuh"
#include "combine_impl.cuh"
#include "gram_impl.cuh"
#include "solver.cuh"

namespace bkmoo {

constexpr int kStreamGramWarps = 8;       // kThreads threads: the Gram pass's thread layout
constexpr int kStreamCombWarps = 4;       // one per tensor-memory lane quadrant
constexpr int kStreamWarps = kStreamGramWarps + kStreamCombWarps + 4;
constexpr uint64_t kStreamWaitNs = 2000000000ull;   // waits for other CTAs give up after 2 s
constexpr uint64_t kStreamLocalNs = 6000000000ull;  // waits within the CTA after 6 s

// items (one 16-byte vector of each gradient for each of the 256 Gram
// threads) per stage, so that a stage is 20-32 KiB
__host__ __device__ constexpr int stream_items(int K) {
  return K == 1 ? 8 : K == 2 ? 4 : K <= 4 ? 2 : 1;
}
__host__ __device__ constexpr int stream_stage_bytes(int K) {
  return K * stream_items(K) * kThreads * 16;
}
// The combination reads again in half stages (10-16 KiB), so that its
// smaller share of the shared memory keeps enough copies in flight.
__host__ __device__ constexpr int stream_half_vecs(int K) { return stream_items(K) * kThreads / 2; }
__host__ __device__ constexpr int stream_gram_buffers(int K) {
  return 128 * 1024 / stream_stage_bytes(K);
}
__host__ __device__ constexpr int stream_comb_buffers(int K) {
  return 80 * 1024 / (stream_stage_bytes(K) / 2);
}
__host__ __device__ constexpr int stream_ring_bytes(int K) {
  return stream_gram_buffers(K) * stream_stage_bytes(K) +
         stream_comb_buffers(K) * (stream_stage_bytes(K) / 2);
}
// tensor-memory slots: 512 columns in two halves (Gram warps 0-3 and 4-7),
// a slot is one stage's K x items x 4 words of every thread
__host__ __device__ constexpr int stream_tmem_slots(int K) { return 64 / (K * stream_items(K)); }
__host__ __device__ constexpr int stream_smem_bytes(int K) {
  return stream_ring_bytes(K) + 128;
}

// ---- tensor memory -------------------------------------------------------------

__device__ __forceinline__ void tmem_st4(uint32_t a, const uint4& x) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x.x),
               "r"(x.y), "r"(x.z), "r"(x.w)
               : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t a, uint4& x) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Words handed from one CTA to another: written once, 0 until then, so a
// reader that finds a word other than 0 has its value.  A partial is stored
// with its bits inverted (only the NaN of all ones would read as unwritten,
// and it is replaced by another NaN), a coefficient below a 1 in bit 32.
__device__ __forceinline__ void st_word(uint64_t* p, uint64_t w) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ uint64_t ld_word(const uint64_t* p) {
  uint64_t w;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ void st_row(uint64_t* p, double x) {
  const uint64_t w = ~(uint64_t)__double_as_longlong(x);
  st_word(p, w ? w : ~0x7ff8000000000000ull);
}
__device__ __forceinline__ double row_value(uint64_t w) { return __longlong_as_double((long long)~w); }
__device__ __forceinline__ void st_beta(uint64_t* p, float x) {
  st_word(p, ((uint64_t)1 << 32) | __float_as_uint(x));
}

// ---- per-chunk geometry ------------------------------------------------------

struct StreamChunk {
  int64_t s, vs, ve, e;  // chunk elements [s, e), aligned vectors [vs, ve)
  int32_t nv, b;         // 16-byte vectors, bucket
};

// What the geometry of a bucket's chunks is computed from.
struct StreamRaw {
  int64_t o0, o1, c0;
  int32_t b;
};
__device__ __forceinline__ StreamRaw stream_raw(const StreamView& sv, int b) {
  StreamRaw r;
  r.b = b;
  r.o0 = __ldg(sv.v.offsets + r.b);
  r.o1 = __ldg(sv.v.offsets + r.b + 1);
  r.c0 = __ldg(sv.v.chunk_prefix + r.b);
  return r;
}
template <int EPV>
__device__ __forceinline__ StreamChunk stream_chunk(const StreamView& sv, const StreamRaw& r,
                                                    int64_t w) {
  StreamChunk c;
  c.s = r.o0 + (w - r.c0) * sv.v.chunk_elems;
  c.e = min(c.s + sv.v.chunk_elems, r.o1);
  c.vs = (c.s + EPV - 1) / EPV * EPV;
  if (c.vs > c.e) c.vs = c.e;
  c.ve = c.e / EPV * EPV;
  if (c.ve < c.vs) c.ve = c.vs;
  c.nv = (int)((c.ve - c.vs) / EPV);
  c.b = r.b;
  return c;
}

// ---- shared state ------------------------------------------------------------

constexpr int kStreamMaxBuf = 16;
constexpr int kStreamDesc = 32;     // Gram chunk descriptors in flight
constexpr int kStreamRed = 3;       // chunks whose triangles await the row warp
constexpr int kStreamLq = 128;      // stages with an L2 claim in flight

constexpr int kStreamSolveWarps = kStreamWarps;   // of a solver CTA: all of them

// A solver team's state (dynamic shared memory of a solver CTA).
template <int K>
struct StreamTeam {
  double t8[2][8 * tri(K)];
  double g8[8 * tri(K)];
  double G[K * K];
  double beta[K];
  float Gf[K * K + (K & 1)];
};

template <int K>
struct StreamShared {
  uint64_t gfull[kStreamMaxBuf], gempty[kStreamMaxBuf];
  uint64_t cfull[kStreamMaxBuf], cempty[kStreamMaxBuf];
  uint64_t tempty[32];
  uint64_t redfull[kStreamRed], redempty[kStreamRed];
  int gkind[kStreamMaxBuf];            // tensor-memory slot of a Gram stage, or -1
  volatile uint32_t tseq[32];          // stage held by each tensor-memory slot
  volatile uint32_t lq[kStreamLq];     // stages with an L2 claim, in order
  uint4 passed;                        // by the combination producer: stages, of those held
                                       // in tensor memory, claimed in L2; its bucket
  StreamChunk gdesc[kStreamDesc];
  float red[kStreamRed][kStreamGramWarps][tri(K)];
  uint32_t tmem;
  volatile int abort;
  volatile int rows_done;      // chunks whose partials this CTA has published
};

// Whole-warp wait for a barrier of this CTA; the result is the same on every
// lane.  False once the kernel gives up.
template <int K>
__device__ __forceinline__ bool stream_wait(StreamShared<K>& sh, const StreamView& sv,
                                            uint64_t* bar, unsigned parity) {
  uint64_t t0 = 0;
  for (unsigned it = 0;; ++it) {
    if (__all_sync(0xffffffffu, bar_try(bar, parity))) return true;
    if ((it & 63u) == 63u) {
      const uint64_t t = stream_ns();
      if (t0 == 0) t0 = t;
      const bool late = t - t0 > kStreamLocalNs;
      if (late) {
        sh.abort = 1;
        record_error(sv.v.hdr, BKMOO_ERR_TIMEOUT);
      }
      if (__any_sync(0xffffffffu, late || sh.abort != 0)) return false;
    }
  }
}

// After a poll of another CTA's data that found nothing: false (on every
// lane) once the wait has to end.
template <int K>
__device__ __forceinline__ bool stream_poll_on(StreamShared<K>& sh, const StreamView& sv,
                                               unsigned it, uint64_t& t0) {
  if ((it & 31u) != 31u) return true;
  const uint64_t t = stream_ns();
  if (t0 == 0) t0 = t;
  const bool late = t - t0 > kStreamWaitNs;
  if (late) {
    record_error(sv.v.hdr, BKMOO_ERR_TIMEOUT);
    *(volatile int32_t*)sv.give_up = 1;
  }
  if (late || *(volatile int32_t*)sv.give_up != 0) sh.abort = 1;
  return !__any_sync(0xffffffffu, sh.abort != 0);
}

// ---- the warps -----------------------------------------------------------------

// A producer's position in the CTA's chunks (the same on every lane).  The
// geometry of chunk i + 1 and the bucket of chunk i + 2 are loaded while
// chunk i is issued, so no copy waits for a chain of global loads.
template <int K, int DT>
struct StreamCursor {
  static constexpr int EPV = elems_per_vec(DT);
  static constexpr int SV = stream_items(K) * kThreads;  // vectors of a stage
  int64_t w;          // chunk i
  int64_t off;        // byte offset of the next stage in every gradient
  int i, n_own;       // index of the chunk in the CTA, number of chunks
  int left;           // vectors of the chunk not yet issued
  int stages;         // stages of the chunk not yet issued
  StreamChunk c;
  StreamRaw next;
  int b2;
  __device__ void begin(const StreamView& sv, int n) {
    n_own = n;
    w = sv.w0 + blockIdx.x;
    next = stream_raw(sv, __ldg(sv.chunk_bucket + w));
    b2 = n > 1 ? __ldg(sv.chunk_bucket + w + sv.n_stream) : 0;
    i = -1;
    w -= sv.n_stream;
    open(sv);
  }
  // false past the last chunk
  __device__ bool open(const StreamView& sv) {
    if (++i >= n_own) return false;
    w += sv.n_stream;
    c = stream_chunk<EPV>(sv, next, w);
    if (i + 1 < n_own) next = stream_raw(sv, b2);
    if (i + 2 < n_own) b2 = __ldg(sv.chunk_bucket + w + 2 * (int64_t)sv.n_stream);
    left = c.nv;
    stages = left > SV ? (left + SV - 1) / SV : 1;
    off = c.vs * (16 / EPV);
    return true;
  }
  // One lane announces the bytes of the next N vectors and copies the K
  // pieces.
  template <int N>
  __device__ __forceinline__ void issue(const GradPtrs& g, unsigned char* dst, uint64_t* full,
                                        uint64_t pol) {
    const unsigned bytes = left > 0 ? (unsigned)(left < N ? left : N) * 16u : 0u;
    if (elect_one()) {
      bar_arrive_tx(full, bytes * K);
      if (bytes) {
#pragma unroll
        for (int k = 0; k < K; ++k)
          bulk_load(dst + k * (N * 16), static_cast<const char*>(g.p[k]) + off, bytes, full, pol);
      }
    }
    skip<N>();
  }
  template <int N>
  __device__ __forceinline__ void skip() {
    left -= N;
    off += N * 16;
  }
};

// Every copy a producer issued into a ring of n slots has landed (before the
// CTA may end; already so unless the kernel gave up).
__device__ __forceinline__ void stream_landed(uint64_t* full, int n, uint32_t issued) {
  for (int i = 0; i < n && (uint32_t)i < issued; ++i) {
    const unsigned par = ((issued - 1 - i) / n) & 1u;  // phase of the slot's last copy
    for (unsigned it = 0; it < 4000000u && !bar_try(full + i, par); ++it) {
    }
  }
}

// Gram producer: copies every stage of the CTA's chunks into the Gram ring
// and decides where its combination will find it again.
template <int K, int DT>
__device__ void stream_gram_producer(StreamShared<K>& sh, unsigned char* gbuf, const GradPtrs& g,
                                     const StreamView& sv, int n_own, int lane) {
  constexpr int SB = stream_stage_bytes(K);
  constexpr int NG = stream_gram_buffers(K), TS = stream_tmem_slots(K);
  const uint64_t pol_first = stream_policy(false), pol_last = stream_policy(true);
  const unsigned lmax = sv.l2_stages, lead = sv.lead;
  StreamCursor<K, DT> q;
  q.begin(sv, n_own);
  uint32_t seq = 0;
  int slot = 0, tslot = 0;
  unsigned par = 1, tpar = 1, tissued = 0, lissued = 0;
  do {
    if (lane == 0) sh.gdesc[q.i % kStreamDesc] = q.c;
    do {
      if (!stream_wait(sh, sv, &sh.gempty[slot], par)) goto out;
      // not too far ahead of the combination, except as far as the next
      // bucket (which the combination may be waiting for)
      uint4 pass;
      for (unsigned it = 0;; ++it) {
        pass = ld_shared_volatile(&sh.passed);
        const bool far = seq - pass.x >= lead && q.c.b > (int)pass.w + 1;
        if (!__any_sync(0xffffffffu, far)) break;
        if ((it & 63u) == 63u && __any_sync(0xffffffffu, sh.abort != 0)) goto out;
      }
      const bool tm = __all_sync(0xffffffffu, tissued - pass.y < (unsigned)TS && bar_test(&sh.tempty[tslot], tpar));
      const bool keep = !tm && __all_sync(0xffffffffu, lissued - pass.z < lmax);
      if (lane == 0) {
        sh.gkind[slot] = tm ? tslot : -1;
        if (tm) sh.tseq[tslot] = seq;
        if (keep) sh.lq[lissued % kStreamLq] = seq;
      }
      __syncwarp();
      if (tm) {
        ++tissued;
        if (++tslot == TS) {
          tslot = 0;
          tpar ^= 1;
        }
      }
      if (keep) ++lissued;
      q.template issue<q.SV>(g, gbuf + slot * SB, &sh.gfull[slot], keep ? pol_last : pol_first);
      --q.stages;
      if (++slot == NG) {
        slot = 0;
        par ^= 1;
      }
      ++seq;
    } while (q.stages > 0);
  } while (q.open(sv));
out:
  stream_landed(sh.gfull, NG, seq);
}

// Combination producer: once a chunk's Gram is complete, copies again the
// stages that are not in tensor memory, each as two half stages.
template <int K, int DT>
__device__ void stream_comb_producer(StreamShared<K>& sh, unsigned char* cbuf, const GradPtrs& g,
                                     const StreamView& sv, int n_own, int lane) {
  constexpr int HB = stream_stage_bytes(K) / 2, HV = stream_half_vecs(K);
  constexpr int NC = stream_comb_buffers(K), TS = stream_tmem_slots(K);
  const uint64_t pol = stream_policy(false);
  StreamCursor<K, DT> q;
  q.begin(sv, n_own);
  uint32_t seq = 0, issued = 0;
  int slot = 0, th = 0;
  unsigned par = 1, tpassed = 0, lpassed = 0;
  do {
    for (unsigned it = 0; __any_sync(0xffffffffu, sh.rows_done <= q.i); ++it)
      if ((it & 63u) == 63u && __any_sync(0xffffffffu, sh.abort != 0)) goto out;
    __threadfence_block();
    do {
      if (__all_sync(0xffffffffu, sh.tseq[th] == seq)) {
        if (++th == TS) th = 0;
        ++tpassed;
        q.template skip<q.SV>();
      } else {
        if (__all_sync(0xffffffffu, sh.lq[lpassed % kStreamLq] == seq)) ++lpassed;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (!stream_wait(sh, sv, &sh.cempty[slot], par)) goto out;
          q.template issue<HV>(g, cbuf + slot * HB, &sh.cfull[slot], pol);
          ++issued;
          if (++slot == NC) {
            slot = 0;
            par ^= 1;
          }
        }
      }
      --q.stages;
      ++seq;
      if (lane == 0)
        st_shared_volatile(&sh.passed, make_uint4(seq, tpassed, lpassed, (uint32_t)q.c.b));
    } while (q.stages > 0);
  } while (q.open(sv));
out:
  stream_landed(sh.cfull, NC, issued);
}

// Gram warps: the chunk's triangle, thread layout and order of
// gram_partials_kernel.
template <int K, int DT>
__device__ void stream_gram(StreamShared<K>& sh, const unsigned char* buf, const GradPtrs& g,
                            const StreamView& sv, int n_own) {
  constexpr int P = tri(K);
  constexpr int U = stream_items(K), SV = U * kThreads;
  constexpr int SB = stream_stage_bytes(K);
  constexpr int NG = stream_gram_buffers(K);
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const uint32_t tm = sh.tmem + ((uint32_t)(wid & 3) << 21) + (uint32_t)(wid >> 2) * 256u;
  int slot = 0;
  unsigned par = 0;
  for (int i = 0; i < n_own; ++i) {
    float acc[P];
#pragma unroll
    for (int p = 0; p < P; ++p) acc[p] = 0.0f;
    int n = 1, nv = 0, nh = 0, nt = 0;
    int64_t sc = 0;
    float xs[K];
    for (int s = 0; s < n; ++s) {
      if (!stream_wait(sh, sv, &sh.gfull[slot], par)) return;
      if (s == 0) {
        const StreamChunk& c = sh.gdesc[i % kStreamDesc];
        nv = c.nv;
        n = nv > SV ? (nv + SV - 1) / SV : 1;
        nh = (int)(c.vs - c.s);
        nt = (int)(c.e - c.ve);
        // the unaligned elements: loaded now, added after the vectors
        if (t < nh + nt) {
          sc = t < nh ? c.s + t : c.ve + (t - nh);
#pragma unroll
          for (int k = 0; k < K; ++k) xs[k] = load_scalar<DT>(g.p[k], sc);
        }
      }
      const int kind = sh.gkind[slot];
      const unsigned char* sb = buf + slot * SB + t * 16;
      if (kind >= 0) tmem_fence_after();
#pragma unroll
      for (int u = 0; u < U; ++u) {
        uint4 r[K];
#pragma unroll
        for (int k = 0; k < K; ++k)
          r[k] = *reinterpret_cast<const uint4*>(sb + (k * U + u) * (kThreads * 16));
        if (u == U - 1) {
          __syncwarp();
          if (lane == 0) bar_arrive(&sh.gempty[slot]);
        }
        if ((s * U + u) * kThreads + t < nv) gram_accumulate<K, DT>(acc, r);
        if (kind >= 0) {
          __syncwarp();
#pragma unroll
          for (int k = 0; k < K; ++k)
            tmem_st4(tm + (uint32_t)(kind * (K * U * 4) + (u * K + k) * 4), r[k]);
        }
      }
      if (++slot == NG) {
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
    __syncwarp();
    tmem_wait_st();
    tmem_fence_before();
    const int rb = i % kStreamRed;
    if (!stream_wait(sh, sv, &sh.redempty[rb], ((unsigned)(i / kStreamRed) & 1u) ^ 1u)) return;
#pragma unroll
    for (int p = 0; p < P; ++p) {
      float v = acc[p];
      v += __shfl_down_sync(0xffffffffu, v, 16);
      v += __shfl_down_sync(0xffffffffu, v, 8);
      v += __shfl_down_sync(0xffffffffu, v, 4);
      v += __shfl_down_sync(0xffffffffu, v, 2);
      v += __shfl_down_sync(0xffffffffu, v, 1);
      if (lane == 0) sh.red[rb][wid][p] = v;
    }
    __syncwarp();
    if (lane == 0) bar_arrive(&sh.redfull[rb]);
  }
}

// The tree over the eight sums; entry p ends in t8[p].
template <int K>
__device__ __forceinline__ void stream_tree8(double* t8, const double (&acc)[(8 * tri(K) + 31) / 32],
                                             int lane) {
  constexpr int P = tri(K), A = (8 * P + 31) / 32;
#pragma unroll
  for (int a = 0; a < A; ++a)
    if (lane + 32 * a < 8 * P) t8[lane + 32 * a] = acc[a];
  __syncwarp();
  for (int p = lane; p < P; p += 32) {
    const double* t = t8 + p;
    const double s = ((t[0] + t[P]) + (t[2 * P] + t[3 * P])) +
                     ((t[4 * P] + t[5 * P]) + (t[6 * P] + t[7 * P]));
    t8[p] = s;                         // entry p is read by this lane only
  }
  __syncwarp();
}

// Row warp: a chunk's partials, the sums over the Gram warps.  `withhold`
// (BKMOO_FLAG_TEST_WITHHOLD_EXCHANGE, CTA 0): those of the first chunk are
// never published, so the solver's wait for them runs out.
template <int K>
__device__ void stream_rows(StreamShared<K>& sh, const StreamView& sv, int n_own, bool withhold,
                            int lane) {
  constexpr int P = tri(K), R = stream_row_words(K);
  for (int i = 0; i < n_own; ++i) {
    const int rb = i % kStreamRed;
    if (!stream_wait(sh, sv, &sh.redfull[rb], (unsigned)(i / kStreamRed) & 1u)) return;
    uint64_t* row = sv.rows + (blockIdx.x + (int64_t)i * sv.n_stream) * R;
    for (int p = lane; p < P; p += 32) {
      double s = 0.0;
#pragma unroll
      for (int q = 0; q < kStreamGramWarps; ++q) s += (double)sh.red[rb][q][p];
      if (!(withhold && i == 0)) st_row(row + p, s);
    }
    __syncwarp();
    if (lane == 0) {
      bar_arrive(&sh.redempty[rb]);
      __threadfence_block();
      sh.rows_done = i + 1;
    }
  }
}

// The set of m rows (at most kSetChunks) at `rows`, as sum_rows8 forms it;
// entry p ends in t8[p].  Lane l keeps the flat entries l, l + 32, ... of
// eight rows.  Waits for words that are not written yet (all loads of the set
// are in flight together: a poll is one round trip to L2).
template <int K>
__device__ bool stream_set(StreamShared<K>& sh, const StreamView& sv, const uint64_t* rows, int m,
                           double* t8, int lane) {
  constexpr int P = tri(K), R = stream_row_words(K), A = (8 * P + 31) / 32;
  static_assert(kSetChunks == 16, "two rows per interleaved sum");
  double acc[A];
#pragma unroll
  for (int a = 0; a < A; ++a) acc[a] = 0.0;
  bool got = __all_sync(0xffffffffu, sh.abort == 0);
  if (got) {
    uint64_t x[2][A];
    uint64_t t0 = 0;
    for (unsigned it = 0;; ++it) {
      bool ok = true;
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int a = 0; a < A; ++a) {
          const int f = lane + 32 * a, j = 8 * h + f / P;
          x[h][a] = 1;
          if (f < 8 * P && j < m) x[h][a] = ld_word(rows + j * R + f % P);
        }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int a = 0; a < A; ++a) ok &= x[h][a] != 0;
      if (__all_sync(0xffffffffu, ok)) break;
      if (!stream_poll_on(sh, sv, it, t0)) {
        got = false;
        break;
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int a = 0; a < A; ++a)
        if ((lane + 32 * a) / P + 8 * h < m) acc[a] += row_value(x[h][a]);
  }
  stream_tree8<K>(t8, acc, lane);
  return got;
}

// Solver CTAs: teams of sv.team warps (2, 4 or 8), each with every
// n_teams-th bucket.  Warp q of a team sums the sets q, q + team, ... as their
// rows arrive and adds set j's sums to the team's eight interleaved sums; the
// team's first warp adds those, solves and publishes.  (The order is that of
// sum_chunk_rows, and of reduce_bucket over the groups of a large bucket.)
// These SMs do nothing else: next to streaming warps the solve of a K = 4
// bucket takes four times as long.
template <int K>
__device__ void stream_solver_cta(StreamShared<K>& sh, unsigned char* dyn, const StreamView& sv,
                                  const SolveParams& prm, float* out_weights, int32_t* out_status) {
  constexpr int P = tri(K), R = stream_row_words(K);
  const PlanView& v = sv.v;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int tw = sv.team, team = wid / tw, q = wid - team * tw;
  const int per_cta = kStreamSolveWarps / tw;
  const int64_t n_teams = (int64_t)per_cta * (gridDim.x - sv.n_stream);
  // per team: two buffers of eight interleaved sums, eight group sums, G;
  // per warp: a tree's scratch
  StreamTeam<K>* tm = reinterpret_cast<StreamTeam<K>*>(dyn) + team;
  double* scratch = reinterpret_cast<double*>(reinterpret_cast<StreamTeam<K>*>(dyn) +
                                              kStreamSolveWarps) + (size_t)wid * (8 * P);
  unsigned turn = 0;
  for (int64_t b = v.b_lo + (blockIdx.x - sv.n_stream) * per_cta + team; b < v.b_hi; b += n_teams) {
    const int64_t c0 = v.chunk_prefix[b], n = v.chunk_prefix[b + 1] - c0;
    uint64_t* rows = sv.rows + (c0 - sv.w0) * R;
    const bool large = n > kGroupMinChunks;
    const int64_t span = large ? kGroupChunks : n;
    if (large && q == 0)
      for (int i = lane; i < 8 * P; i += 32) tm->g8[i] = 0.0;
    int64_t grp = 0;
    for (int64_t g0 = 0; g0 < n; g0 += span, ++grp, ++turn) {
      const int64_t m = min(span, n - g0);
      const int sets = (int)((m + kSetChunks - 1) / kSetChunks);
      double* t8 = tm->t8[turn & 1];
      for (int j = q; j < 8; j += tw)
        for (int p = lane; p < P; p += 32) t8[j * P + p] = 0.0;
      __syncwarp();
      for (int s = q; s < sets; s += tw) {
        const int64_t at = (int64_t)s * kSetChunks;
        const int rows_in = (int)min((int64_t)kSetChunks, m - at);
        (void)stream_set(sh, sv, rows + (g0 + at) * R, rows_in, scratch, lane);
        for (int p = lane; p < P; p += 32) t8[(s & 7) * P + p] += scratch[p];
        __syncwarp();
      }
      __threadfence_block();
      asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(tw * 32) : "memory");
      if (q != 0) continue;
      for (int p = lane; p < P; p += 32) {
        const double* t = t8 + p;
        const double s = ((t[0] + t[P]) + (t[2 * P] + t[3 * P])) +
                         ((t[4 * P] + t[5 * P]) + (t[6 * P] + t[7 * P]));
        if (large) tm->g8[(grp & 7) * P + p] += s;
        else tm->g8[p] = s;
      }
      __syncwarp();
    }
    if (q != 0) continue;
    if (__any_sync(0xffffffffu, sh.abort != 0)) continue;
    for (int p = lane; p < P; p += 32) {
      const double* t = tm->g8 + p;
      const double s = large ? ((t[0] + t[P]) + (t[2 * P] + t[3 * P])) +
                                   ((t[4 * P] + t[5 * P]) + (t[6 * P] + t[7 * P]))
                             : t[0];
      int i = 0, r = p;
      while (r >= K - i) {
        r -= K - i;
        ++i;
      }
      tm->G[i * K + i + r] = s;
      tm->G[(i + r) * K + i] = s;
    }
    __syncwarp();
    const int st = solver::solve_bucket_warp<K>(K, tm->G, tm->Gf, prm, b, tm->beta, lane);
    // BKMOO_FLAG_TEST_WITHHOLD: the first bucket's coefficients are never
    // published, so the waits for them run out (the failure-detection test)
    const bool withhold = b == v.b_lo && (prm.flags & BKMOO_FLAG_TEST_WITHHOLD);
    if (lane < K) {
      const float f = (float)tm->beta[lane];
      if (!withhold) st_beta(rows + P + lane, f);
      v.beta[b * K + lane] = f;
      if (out_weights) out_weights[b * K + lane] = f;
    }
    if (lane == 0 && out_status) out_status[b] = st;
    __syncwarp();
  }
}

// d = sum_k beta_k x_k of one vector position, k ascending; two elements per
// paired fp32 FMA, each rounded as fmaf rounds it.
template <int K, int DT>
__device__ __forceinline__ void stream_combine_vec(const uint4 (&r)[K], const float (&beta)[K],
                                                   void* out, int dto, int64_t el) {
  constexpr int EPV = elems_per_vec(DT);
  float y[EPV];
#pragma unroll
  for (int q = 0; q < EPV; q += 2) {
    float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < K; ++k)
      s = __ffma2_rn(make_float2(beta[k], beta[k]),
                     make_float2(vec_elem<DT>(r[k], q), vec_elem<DT>(r[k], q + 1)), s);
    y[q] = s.x;
    y[q + 1] = s.y;
  }
  if (dto == BKMOO_F32) store_out<BKMOO_F32>(out, el, y, EPV);
  else store_out<BKMOO_BF16>(out, el, y, EPV);
}

// Combination warps: thread t has the vector positions of the Gram threads t and
// t + 128.
template <int K, int DT>
__device__ void stream_combine(StreamShared<K>& sh, const unsigned char* cbuf, const GradPtrs& g,
                               const StreamView& sv, void* out, int dto, int n_own) {
  constexpr int EPV = elems_per_vec(DT);
  constexpr int U = stream_items(K), SV = U * kThreads;
  constexpr int HB = stream_stage_bytes(K) / 2, HV = stream_half_vecs(K);
  constexpr int NC = stream_comb_buffers(K);
  constexpr int TS = stream_tmem_slots(K);
  constexpr int CT = 32 * kStreamCombWarps;
  static_assert(HV % CT == 0, "a half stage is whole positions of every combination thread");
  static_assert(kThreads == 2 * CT, "two Gram threads' positions per combination thread");
  const int ct = threadIdx.x - kThreads, lane = ct & 31, c = ct >> 5;
  const uint32_t tm = sh.tmem + ((uint32_t)c << 21);
  uint32_t seq = 0;
  int slot = 0, th = 0;
  unsigned par = 0;
  const int64_t w0 = sv.w0 + blockIdx.x;
  StreamRaw next = stream_raw(sv, __ldg(sv.chunk_bucket + w0));
  int b2 = n_own > 1 ? __ldg(sv.chunk_bucket + w0 + sv.n_stream) : 0;
  int prev = -1;
  float beta[K];
  for (int i = 0; i < n_own; ++i) {
    const int64_t w = w0 + (int64_t)i * sv.n_stream;
    const StreamChunk d = stream_chunk<EPV>(sv, next, w);
    if (d.b != prev) {      // wait for the bucket's coefficients
      prev = d.b;
      const uint64_t* words =
          sv.rows + (next.c0 - sv.w0) * stream_row_words(K) + tri(K);
      uint64_t x = 0;
      uint64_t t0 = 0;
      for (unsigned it = 0;; ++it) {
        if (lane < K) x = ld_word(words + lane);
        if (__all_sync(0xffffffffu, lane >= K || x != 0)) break;
        if (!stream_poll_on(sh, sv, it, t0)) return;
      }
#pragma unroll
      for (int k = 0; k < K; ++k) beta[k] = __uint_as_float(__shfl_sync(0xffffffffu, (uint32_t)x, k));
    }
    // the chunk's own Gram stages (and what they left in tensor memory) are
    // ordered before its combination
    while (__shfl_sync(0xffffffffu, sh.rows_done, 0) <= i)
      if (__any_sync(0xffffffffu, sh.abort != 0)) return;
    __threadfence_block();
    if (i + 1 < n_own) next = stream_raw(sv, b2);
    if (i + 2 < n_own) b2 = __ldg(sv.chunk_bucket + w + 2 * (int64_t)sv.n_stream);
    const int n = d.nv > SV ? (d.nv + SV - 1) / SV : 1;
    const int nh = (int)(d.vs - d.s), nt = (int)(d.e - d.ve);
    const int64_t sc = ct < nh ? d.s + ct : d.ve + (ct - nh);
    float xs[K];
    if (ct < nh + nt) {
#pragma unroll
      for (int k = 0; k < K; ++k) xs[k] = load_scalar<DT>(g.p[k], sc);
    }
    __syncwarp();
    for (int s = 0; s < n; ++s, ++seq) {
      const bool held = sh.tseq[th] == seq;
      if (held) {
        tmem_fence_after();
        // warp c reads both column halves: those of Gram warps c and c + 4
        constexpr int N = 2 * U;
        uint4 r[N][K];
#pragma unroll
        for (int u = 0; u < N; ++u)
#pragma unroll
          for (int k = 0; k < K; ++k)
            tmem_ld4(tm + (uint32_t)(u & 1) * 256u +
                         (uint32_t)(th * (K * U * 4) + (u / 2 * K + k) * 4),
                     r[u][k]);
        tmem_wait_ld();
        tmem_fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(&sh.tempty[th]);
#pragma unroll
        for (int u = 0; u < N; ++u) {
          const int v0 = s * SV + u * CT + ct;
          if (v0 < d.nv) stream_combine_vec<K, DT>(r[u], beta, out, dto, d.vs + (int64_t)v0 * EPV);
        }
        __syncwarp();
        if (++th == TS) th = 0;
      } else {
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          if (!stream_wait(sh, sv, &sh.cfull[slot], par)) return;
          const unsigned char* sb = cbuf + slot * HB + ct * 16;
          constexpr int N = HV / CT;
          uint4 r[N][K];
#pragma unroll
          for (int u = 0; u < N; ++u)
#pragma unroll
            for (int k = 0; k < K; ++k)
              r[u][k] = *reinterpret_cast<const uint4*>(sb + (k * HV + u * CT) * 16);
          __syncwarp();
          if (lane == 0) bar_arrive(&sh.cempty[slot]);
#pragma unroll
          for (int u = 0; u < N; ++u) {
            const int v0 = s * SV + h * HV + u * CT + ct;
            if (v0 < d.nv)
              stream_combine_vec<K, DT>(r[u], beta, out, dto, d.vs + (int64_t)v0 * EPV);
          }
          __syncwarp();
          if (++slot == NC) {
            slot = 0;
            par ^= 1;
          }
        }
      }
    }
    if (ct < nh + nt) {
      float y = 0.0f;
#pragma unroll
      for (int k = 0; k < K; ++k) y = fmaf(beta[k], xs[k], y);
      if (dto == BKMOO_F32) store_scalar<BKMOO_F32>(out, sc, y);
      else store_scalar<BKMOO_BF16>(out, sc, y);
    }
  }
}

// grid: n_stream + n_solve CTAs, cooperative launch.
template <int K, int DT>
__global__ void __launch_bounds__(32 * kStreamWarps, 1)
    stream_resolve_kernel(const GradPtrs g, const StreamView sv, const SolveParams prm,
                          float* out_weights, int32_t* out_status, void* out, int dto) {
  __shared__ __align__(16) StreamShared<K> sh;
  extern __shared__ unsigned char st_dyn[];
  // uniform across the grid: every CTA leaves before any barrier
  if (!header_ok(sv.v)) {
    if (blockIdx.x == 0) {
      if (threadIdx.x == 0) {
        if (sv.reset) sv.v.hdr->status = BKMOO_ERR_WORKSPACE;
        else record_error(sv.v.hdr, BKMOO_ERR_WORKSPACE);
      }
      if (out_status)
        for (int64_t b = sv.v.b_lo + threadIdx.x; b < sv.v.b_hi; b += blockDim.x)
          out_status[b] = BKMOO_ERR_WORKSPACE;
    }
    return;
  }
  if (sv.reset && blockIdx.x == 0 && threadIdx.x == 0) sv.v.hdr->status = BKMOO_OK;
  unsigned char* buf = reinterpret_cast<unsigned char*>(
      ((uintptr_t)st_dyn + 127) & ~(uintptr_t)127);
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int CW = kStreamCombWarps, kP = kStreamGramWarps + CW;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStreamMaxBuf; ++i) {
      bar_init(&sh.gfull[i], 1);
      bar_init(&sh.gempty[i], kStreamGramWarps);
      bar_init(&sh.cfull[i], 1);
      bar_init(&sh.cempty[i], CW);
    }
    for (int i = 0; i < 32; ++i) {
      bar_init(&sh.tempty[i], CW);
      sh.tseq[i] = 0xffffffffu;
    }
    for (int i = 0; i < kStreamLq; ++i) sh.lq[i] = 0xffffffffu;
    sh.passed = make_uint4(0u, 0u, 0u, (uint32_t)sv.v.b_lo);
    for (int i = 0; i < kStreamRed; ++i) {
      bar_init(&sh.redfull[i], kStreamGramWarps);
      bar_init(&sh.redempty[i], 1);
    }
    sh.abort = 0;
    sh.rows_done = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (blockIdx.x >= (unsigned)sv.n_stream) {
    __syncthreads();
    stream_solver_cta<K>(sh, buf, sv, prm, out_weights, out_status);
    return;
  }
  if (wid == kP + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     st_smem(&sh.tmem))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    tmem_fence_before();
  }
  __syncthreads();
  tmem_fence_after();
  const int n_own = (int)((sv.v.c_hi - sv.w0 - blockIdx.x + sv.n_stream - 1) / sv.n_stream);
  unsigned char* cbuf = buf + stream_gram_buffers(K) * stream_stage_bytes(K);
  if (wid < kStreamGramWarps) stream_gram<K, DT>(sh, buf, g, sv, n_own);
  else if (wid < kP) stream_combine<K, DT>(sh, cbuf, g, sv, out, dto, n_own);
  else if (wid == kP) stream_gram_producer<K, DT>(sh, buf, g, sv, n_own, lane);
  else if (wid == kP + 1) stream_rows<K>(
        sh, sv, n_own, blockIdx.x == 0 && (prm.flags & BKMOO_FLAG_TEST_WITHHOLD_EXCHANGE), lane);
  else if (wid == kP + 2) stream_comb_producer<K, DT>(sh, cbuf, g, sv, n_own, lane);
  // A Gram warp that gives up leaves its chunk's tensor-memory stores in
  // flight; none may be when the memory is handed back.
  __syncwarp();
  tmem_wait_st();
  tmem_wait_ld();
  tmem_fence_before();
  __syncthreads();
  if (wid == kP + 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(sh.tmem));
}

}  // namespace bkmoo
