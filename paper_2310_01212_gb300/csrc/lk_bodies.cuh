/*
 * lk_bodies.cuh -- the work a descriptor names (Sec. I: "a descriptor of the
 * work and a reference to the in/out data items"), split across the S CTAs
 * of a cluster.  CTA `r` of S takes a contiguous, 16-byte-aligned share of
 * the data; the split depends only on (n, S), so a result does not depend on
 * which descriptors ran before or beside it.
 *
 * Streaming bodies (add, copy, sum, histogram) move a CTA's share through
 * shared memory: thread 0 issues TMA bulk copies (cp.async.bulk, 16-byte
 * granules, completion counted on an mbarrier per stage) into a ring of
 * LK_STAGES stages, so up to three stages (96 KB) per SM are in flight while
 * every warp consumes the fourth; registers no longer bound the bytes in
 * flight.  One CTA barrier per chunk both releases the consumed stage for
 * refill and makes every thread agree on whether the stage arrived in time.
 *
 * Bodies:
 *   add_i32   out[i] = a[i] + b[i] mod 2^32: both inputs staged, 128-bit
 *             streaming stores of the sums
 *   copy_i32  out[i] = in[i]: staged in, then a bulk store straight from the
 *             stage (no registers touched)
 *   hist_u8   per-CTA counts -> added to the output (global atomics) once rank
 *             0 has cleared it; split parts and ordinary launches go through an
 *             accumulator.  Small shares count into per-warp bins with
 *             shared atomics; shares from 16 KB count into lane-private
 *             32-bit counters, which no two lanes of a warp ever share, so
 *             random bytes cause no shared-memory bank conflicts; with one
 *             CTA per SM every warp streams its part through a ring of its own.
 *   sum_f32   per-thread float accumulators, warp shuffles, per-CTA partial;
 *             rank 0 adds the partials in rank order in binary64
 *   gemm64    64x64x64 float32 tiles staged into shared memory by TMA bulk
 *             copies.  Whole tiles (one CTA per SM, 256 threads): tcgen05
 *             tensor cores on split-bf16 operands, or (on request, or with
 *             two CTAs per SM) packed FFMA in k order, four tiles at a time
 *             (two).  Row blocks of split tiles and other block sizes: 4x4
 *             register micro-tiles, FFMA in k order
 * Used by the persistent kernel and by the ordinary-launch baseline kernels.
 */
#ifndef LK_BODIES_CUH
#define LK_BODIES_CUH
#include "lk_device.cuh"
#include "lk_layout.h"

namespace lk {

/* Contiguous share [beg, end) of `units` for rank r of S. */
__device__ __forceinline__ void share(uint64_t units, int r, int S, uint64_t& beg, uint64_t& end) {
  beg = units * (uint64_t)r / (uint64_t)S;
  end = units * (uint64_t)(r + 1) / (uint64_t)S;
}

__device__ __forceinline__ int4 add4(int4 x, int4 y) {
  return make_int4((int)((unsigned)x.x + (unsigned)y.x), (int)((unsigned)x.y + (unsigned)y.y),
                   (int)((unsigned)x.z + (unsigned)y.z), (int)((unsigned)x.w + (unsigned)y.w));
}

/* ---- shared-memory layout of a CTA ------------------------------------- */
/* With one CTA per SM (P = 1) the streaming bodies use 192 KB of the CTA's
 * 224 KB: a 64 KB work region (histogram counters) and a 128 KB ring of
 * LK_STAGES streaming stages; the FFMA GEMM's stages span those 192 KB and
 * the tensor-core GEMM uses all 224 KB (LK_TC_SMEM).  With two CTAs per SM
 * (P = 2) each CTA owns half of every region, so the bytes in flight per SM
 * stay the same. */
#define LK_SMEM_WORK (64u * 1024u)     /* histogram counters or GEMM stages   */
#define LK_SMEM_STREAM (128u * 1024u)  /* streaming stages                    */
#define LK_SMEM_DYN (LK_SMEM_WORK + LK_SMEM_STREAM)
#define LK_GEMM_STAGE_FLOATS 8192u     /* one GEMM stage: A rows 16 KB + B tile 16 KB */
#define LK_HIST_COPIES 1u              /* lane-private counter copies (32 KB each) */
#define LK_NUM_BARS 8u                 /* mbarriers: one per stage; the tensor-core GEMM's MMA completion in 4, 5 */
#define LK_WARP_BARS (32u * LK_STAGES)  /* then one per stage of each warp's own ring (histogram) */
#define LK_ALL_BARS (LK_NUM_BARS + LK_WARP_BARS)

template <int P>
struct SmemCfg {
  static_assert(P == 1 || P == 2, "one or two CTAs per SM");
  static constexpr uint32_t work_bytes = LK_SMEM_WORK / P;
  static constexpr uint32_t stream_bytes = LK_SMEM_STREAM / P;
  static constexpr uint32_t dyn_bytes = work_bytes + stream_bytes;
  static constexpr uint32_t gemm_stages = dyn_bytes / (LK_GEMM_STAGE_FLOATS * 4u);   /* 6 or 3 */
  static constexpr uint32_t hist_copies = LK_HIST_COPIES;
  static_assert(gemm_stages <= LK_NUM_BARS, "one mbarrier per stage");
};

/* Time limits of one body.  Every staging wait ends by `deadline`.  A
 * non-zero `rate` (bytes per microsecond for this CTA) paces the TMA loads:
 * a token bucket as deep as the stage ring, so the first stages load at once
 * and each later one no earlier than its bytes allow; the deadline then
 * moves out by the paced duration of the CTA's share. */
struct Pace {
  uint64_t deadline;
  uint64_t rate;
  const int32_t* gate;   /* non-null: yield to critical descriptors (lk_set_role) */
};

/* Thread 0: sleep until `due` (%globaltimer ns); bounded by `due` itself. */
__device__ __forceinline__ void sleep_until(uint64_t due) {
  for (uint64_t now = gtime(); now < due; now = gtime()) {
    const uint64_t left = due - now;
    __nanosleep(left > 2000u ? 2000u : (uint32_t)left);
  }
}

/* Load yielding of one issuing thread (lk_set_role): before each refill of
 * a stage it holds while the count of running critical descriptors is
 * positive.  The count tested is the one loaded at the previous refill (the
 * load's round trip overlaps the stage wait in between, so a refill never
 * waits on L2 for it); one hold lasts at most LK_YIELD_HOLD_NS and a body's
 * holds together at most LK_YIELD_BUDGET_NS, by which its stage deadline is
 * extended.  The count is a hint: a stale value only shifts a hold by one
 * stage. */
#define LK_YIELD_HOLD_NS 1000000ull
#define LK_YIELD_BUDGET_NS 8000000ull
struct Yield {
  const int32_t* gate;
  int32_t seen;
  uint64_t end;
  __device__ __forceinline__ explicit Yield(const int32_t* g) : gate(g), seen(0), end(0) {
    if (gate) {
      end = gtime() + LK_YIELD_BUDGET_NS;
      seen = ld_relaxed_gpu_s32(gate);
    }
  }
  __device__ __forceinline__ void hold() {
    if (!gate) return;
    if (seen > 0) {
      uint64_t now = gtime();
      const uint64_t lim = now + LK_YIELD_HOLD_NS < end ? now + LK_YIELD_HOLD_NS : end;
      while (now < lim && ld_relaxed_gpu_s32(gate) > 0) {
        __nanosleep(256);
        now = gtime();
      }
    }
    seen = ld_relaxed_gpu_s32(gate);
  }
};

/* Stream the 16-byte vectors [beg, end) of NIN inputs through the stages.
 * consume(v0, nv, s0, s1) runs on every thread for each chunk: vectors
 * v0 .. v0+nv-1 of the share sit at s0[0..nv) (and s1[0..nv) for a second
 * input).  With STORE, consume issues bulk stores from the stage (thread 0)
 * and a stage is refilled only after those stores have read it.  `phase`
 * holds one parity bit per mbarrier and persists across descriptors.
 * Returns false, on every thread alike, if a stage did not arrive before
 * the deadline; this CTA's copies in flight are allowed to land first. */
template <int NIN, bool STORE, int P, class F>
__device__ __forceinline__ bool stream(const uint4* in0, const uint4* in1, uint64_t beg, uint64_t end,
                                       unsigned char* stage_mem, uint64_t* bars, uint32_t& phase, Pace pace,
                                       F&& consume) {
  constexpr uint32_t stage_vec = SmemCfg<P>::stream_bytes / LK_STAGES / NIN / 16u;   /* vectors per input per chunk */
  const uint64_t total = end > beg ? end - beg : 0;
  const uint64_t nch = (total + stage_vec - 1) / stage_vec;
  if (nch == 0) return true;
  constexpr uint64_t chunk_bytes = (uint64_t)stage_vec * 16u * NIN;
  const uint64_t deadline = (pace.rate ? pace.deadline + total * 16u * NIN * 1000u / pace.rate : pace.deadline) +
                            (pace.gate ? LK_YIELD_BUDGET_NS : 0u);
  const uint64_t t_first = pace.rate && threadIdx.x == 0 ? gtime() : 0;
  Yield yield(threadIdx.x == 0 ? pace.gate : nullptr);
  auto sbuf = [&](uint32_t st, int which) {
    return reinterpret_cast<uint4*>(stage_mem + ((size_t)st * NIN + which) * stage_vec * 16u);
  };
  auto issue = [&](uint64_t ch) {   /* thread 0 only */
    const uint32_t st = (uint32_t)(ch % LK_STAGES);
    const uint64_t v0 = beg + ch * stage_vec;
    const uint32_t nv = (uint32_t)((end - v0) < stage_vec ? (end - v0) : stage_vec);
    if (!LK_INB(v0 >= beg && v0 + nv <= end && ((uintptr_t)(in0 + v0) & 15u) == 0 &&
                    (NIN == 1 || ((uintptr_t)(in1 + v0) & 15u) == 0), LK_OOB_STREAM_LOAD) ||
        !LK_INB(((size_t)st * NIN + NIN) * stage_vec * 16u <= SmemCfg<P>::stream_bytes, LK_OOB_STREAM_SMEM)) {
      mbar_expect_tx(&bars[st], 0u);   /* skipped: the phase completes with no bytes */
      return;
    }
    mbar_expect_tx(&bars[st], nv * 16u * NIN);
    bulk_g2s(sbuf(st, 0), in0 + v0, nv * 16u, &bars[st]);
    if (NIN > 1) bulk_g2s(sbuf(st, 1), in1 + v0, nv * 16u, &bars[st]);
  };
  if (threadIdx.x == 0) {
    yield.hold();
    fence_proxy_async_global();   /* earlier generic writes before these async reads */
    fence_proxy_async_smem();     /* earlier generic shared accesses before async writes */
    for (uint64_t ch = 0; ch < nch && ch < LK_STAGES; ++ch) issue(ch);
  }
  for (uint64_t ch = 0; ch < nch; ++ch) {
    const uint32_t st = (uint32_t)(ch % LK_STAGES);
    const bool ok = mbar_wait(&bars[st], (phase >> st) & 1u, deadline);
    if (__syncthreads_or(!ok)) {
      if (threadIdx.x == 0) {
        for (uint64_t c2 = ch; c2 < nch && c2 < ch + LK_STAGES; ++c2) {
          const uint32_t s2 = (uint32_t)(c2 % LK_STAGES);
          mbar_wait(&bars[s2], (phase >> s2) & 1u, deadline + 1000000000ull);
        }
        if (STORE) bulk_wait_all();
      }
      __syncthreads();
      return false;
    }
    phase ^= 1u << st;
    /* every thread has finished chunk ch-1: refill its stage */
    if (threadIdx.x == 0 && ch >= 1 && ch - 1 + LK_STAGES < nch) {
      if (pace.rate) sleep_until(t_first + ch * chunk_bytes * 1000u / pace.rate);
      yield.hold();
      if (STORE) bulk_wait_read_all();
      fence_proxy_async_smem();
      issue(ch - 1 + LK_STAGES);
    }
    const uint64_t v0 = beg + ch * stage_vec;
    const uint32_t nv = (uint32_t)((end - v0) < stage_vec ? (end - v0) : stage_vec);
    consume(v0, nv, sbuf(st, 0), NIN > 1 ? sbuf(st, 1) : nullptr);
  }
  __syncthreads();   /* every consumer is done before a later body reuses the stages */
  if (STORE && threadIdx.x == 0) {
    bulk_wait_all();
    fence_proxy_async_global();   /* the stores' writes before this thread's later release */
  }
  return true;
}

/* Shares of at most K vectors per thread skip the stage ring: every thread
 * issues all of its 128-bit loads at once and then consumes them -- one
 * global round trip, with no TMA issue, mbarrier wait or CTA barrier, which
 * on a share of a few tens of KB cost more than they hide.  f(i, v, x) gets
 * the thread's i-th vector, index v of the input.  Used by the add and sum
 * bodies of kernels with registers to spare (DIRECT: at most 256 threads,
 * one CTA per SM); elsewhere the extra live registers would spill. */
template <int K, class F>
__device__ __forceinline__ void direct(const uint4* in, uint64_t beg, uint64_t total, F&& f) {
  const uint32_t T = blockDim.x;
  uint4 q[K];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const uint64_t v = threadIdx.x + (uint64_t)i * T;
    q[i] = make_uint4(0, 0, 0, 0);
    if (v < total) q[i] = ld_stream(in + beg + v);
  }
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const uint64_t v = threadIdx.x + (uint64_t)i * T;
    if (v < total) f(i, beg + v, q[i]);
  }
}
#define LK_DIRECT_ADD 4u     /* vectors per thread per input: add  */
#define LK_DIRECT_ONE 8u     /* vectors per thread: sum, histogram */

/* ---- int32 add / copy -------------------------------------------------- */
template <int P, bool DIRECT = false>
__device__ __forceinline__ bool body_add(const lk_slot& d, int r, int S, unsigned char* dsm, uint64_t* bars,
                                         uint32_t& phase, Pace pace) {
  const uint64_t n = d.n, nv = n >> 2;
  uint64_t beg, end;
  share(nv, r, S, beg, end);
  if (!LK_INB(beg <= end && end <= nv, LK_OOB_SHARE)) end = beg;
  int4* o = reinterpret_cast<int4*>(d.out);
  const uint32_t T = blockDim.x;
  bool ok = true;
  if (DIRECT && end - beg <= (uint64_t)LK_DIRECT_ADD * T) {
    const int4* a = reinterpret_cast<const int4*>(d.in0);
    const int4* b = reinterpret_cast<const int4*>(d.in1);
    int4 x[LK_DIRECT_ADD], y[LK_DIRECT_ADD];
#pragma unroll
    for (uint32_t i = 0; i < LK_DIRECT_ADD; ++i) {
      const uint64_t v = beg + threadIdx.x + (uint64_t)i * T;
      x[i] = y[i] = make_int4(0, 0, 0, 0);
      if (v < end) {
        x[i] = ld_stream(a + v);
        y[i] = ld_stream(b + v);
      }
    }
#pragma unroll
    for (uint32_t i = 0; i < LK_DIRECT_ADD; ++i) {
      const uint64_t v = beg + threadIdx.x + (uint64_t)i * T;
      if (v < end) st_stream(o + v, add4(x[i], y[i]));
    }
  } else {
    ok = stream<2, false, P>(reinterpret_cast<const uint4*>(d.in0), reinterpret_cast<const uint4*>(d.in1),
                             beg, end, dsm + SmemCfg<P>::work_bytes, bars, phase, pace,
                             [&](uint64_t v0, uint32_t cnt, const uint4* s0, const uint4* s1) {
                               const int4* a = reinterpret_cast<const int4*>(s0);
                               const int4* b = reinterpret_cast<const int4*>(s1);
                               for (uint32_t v = threadIdx.x; v < cnt; v += T)
                                 if (LK_INB(v0 + v < end, LK_OOB_STORE)) st_stream(o + v0 + v, add4(a[v], b[v]));
                             });
  }
  if (r == S - 1) {
    const int32_t* as = reinterpret_cast<const int32_t*>(d.in0);
    const int32_t* bs = reinterpret_cast<const int32_t*>(d.in1);
    int32_t* os = reinterpret_cast<int32_t*>(d.out);
    for (uint64_t j = nv * 4 + threadIdx.x; j < n; j += T) os[j] = (int32_t)((uint32_t)as[j] + (uint32_t)bs[j]);
  }
  return ok;
}

template <int P>
__device__ __forceinline__ bool body_copy(const lk_slot& d, int r, int S, unsigned char* dsm, uint64_t* bars,
                                          uint32_t& phase, Pace pace) {
  const uint64_t n = d.n, nv = n >> 2;
  uint64_t beg, end;
  share(nv, r, S, beg, end);
  if (!LK_INB(beg <= end && end <= nv, LK_OOB_SHARE)) end = beg;
  uint4* o = reinterpret_cast<uint4*>(d.out);
  const bool ok = stream<1, true, P>(reinterpret_cast<const uint4*>(d.in0), nullptr, beg, end, dsm + SmemCfg<P>::work_bytes, bars,
                                  phase, pace, [&](uint64_t v0, uint32_t cnt, const uint4* s0, const uint4*) {
                                    if (threadIdx.x == 0 && LK_INB(v0 + cnt <= end, LK_OOB_STORE)) {
                                      bulk_s2g(o + v0, s0, cnt * 16u);
                                      bulk_commit();
                                    }
                                  });
  if (r == S - 1) {
    const int32_t* as = reinterpret_cast<const int32_t*>(d.in0);
    int32_t* os = reinterpret_cast<int32_t*>(d.out);
    for (uint64_t j = nv * 4 + threadIdx.x; j < n; j += blockDim.x) os[j] = as[j];
  }
  return ok;
}

/* ---- float32 sum: this CTA's partial (valid in thread 0) ---------------- */
template <int P, bool DIRECT = false>
__device__ __forceinline__ bool body_sum(const lk_slot& d, int r, int S, unsigned char* dsm, uint64_t* bars,
                                         uint32_t& phase, Pace pace, float* red, float* partial_out) {
  const uint64_t n = d.n, nv = n >> 2;
  uint64_t beg, end;
  share(nv, r, S, beg, end);
  if (!LK_INB(beg <= end && end <= nv, LK_OOB_SHARE)) end = beg;
  const uint32_t T = blockDim.x;
  float acc0 = 0.f, acc1 = 0.f;
  bool ok = true;
  if (DIRECT && end - beg <= (uint64_t)LK_DIRECT_ONE * T) {
    /* the thread's vectors alternate between the two accumulators, as in
     * the staged loop below over a single chunk */
    direct<LK_DIRECT_ONE>(reinterpret_cast<const uint4*>(d.in0), beg, end - beg, [&](int i, uint64_t, uint4 q) {
      const float4 p = make_float4(__uint_as_float(q.x), __uint_as_float(q.y), __uint_as_float(q.z), __uint_as_float(q.w));
      if (i & 1) acc1 += (p.x + p.y) + (p.z + p.w);
      else acc0 += (p.x + p.y) + (p.z + p.w);
    });
  } else ok = stream<1, false, P>(reinterpret_cast<const uint4*>(d.in0), nullptr, beg, end, dsm + SmemCfg<P>::work_bytes,
                                   bars, phase, pace, [&](uint64_t, uint32_t cnt, const uint4* s0, const uint4*) {
                                     const float4* x = reinterpret_cast<const float4*>(s0);
                                     uint32_t v = threadIdx.x;
                                     for (; v + T < cnt; v += 2 * T) {
                                       const float4 p = x[v], q = x[v + T];
                                       acc0 += (p.x + p.y) + (p.z + p.w);
                                       acc1 += (q.x + q.y) + (q.z + q.w);
                                     }
                                     if (v < cnt) {
                                       const float4 p = x[v];
                                       acc0 += (p.x + p.y) + (p.z + p.w);
                                     }
                                   });
  if (r == S - 1) {
    const float* xs = reinterpret_cast<const float*>(d.in0);
    for (uint64_t j = nv * 4 + threadIdx.x; j < n; j += T) acc0 += xs[j];
  }
  float s = acc0 + acc1;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) red[warp] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (uint32_t w = 0; w < T / 32; ++w) t += red[w];
    *partial_out = t;
  }
  return ok;
}

/* One warp (lanes `lane` 0-31): out[0] = partials added in rank order (binary64). */
__device__ __forceinline__ void combine_sum(const lk_slot& d, const float* partial, int S, uint32_t lane) {
  if (lane >= 32) return;
  double s = 0.0;
  for (int q = (int)lane; q < S; q += 32) s += (double)__ldcg(partial + q);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) *reinterpret_cast<float*>(d.out) = (float)s;
}

/* ---- uint8 histogram ---------------------------------------------------- */
/* Shares below this many bytes per CTA use per-warp bins, whose set-up and
 * read-out are cheap; larger shares use the conflict-free lane-private path
 * (measured crossover on GB300: a 28 KB share counts in 2.2 us lane-private
 * against 2.9 us in per-warp bins; a 7 KB share in 1.9 against 1.7 us). */
#define LK_HIST_SMALL_BYTES (16u * 1024u)

__device__ __forceinline__ void count4_warp(uint32_t* bins, uint32_t w) {
  atomicAdd(&bins[w & 0xffu], 1u);
  atomicAdd(&bins[(w >> 8) & 0xffu], 1u);
  atomicAdd(&bins[(w >> 16) & 0xffu], 1u);
  atomicAdd(&bins[w >> 24], 1u);
}

/* Lane-private counters: word (v << 5) | lane of a copy (8192 words, 32 KB)
 * counts bin v for this lane alone, so lane l only touches bank l, and one
 * byte costs an extract, an address and one shared reduction.  32-bit
 * counters cannot overflow: a share holds fewer than 2^31 bytes. */
__device__ __forceinline__ void count4_lane(uint32_t lane_addr, uint32_t w) {
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const uint32_t v = (w >> (8 * b)) & 0xffu;
    asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], 1;" ::"r"(lane_addr + (v << 7)) : "memory");
  }
}

/* Thread v (< 256) adds bin v over the 32 lanes of every copy.  The loads of
 * a row start at thread-dependent columns, so each 8-thread phase of a
 * 128-bit warp load touches all 32 banks once. */
template <int P>
__device__ __forceinline__ uint32_t hist_readout(const uint32_t* sh, uint32_t v) {
  uint32_t tot = 0;
  for (uint32_t c = 0; c < SmemCfg<P>::hist_copies; ++c) {
    const uint4* rw = reinterpret_cast<const uint4*>(sh + c * 8192u + v * 32u);
#pragma unroll
    for (uint32_t j = 0; j < 8; ++j) {
      const uint4 q = rw[(j + v) & 7u];
      tot += (q.x + q.y) + (q.z + q.w);
    }
  }
  return tot;
}

__device__ __forceinline__ void hist_zero(uint32_t* sh, uint32_t words) {
  uint4* z = reinterpret_cast<uint4*>(sh);
  for (uint32_t i = threadIdx.x; i < words / 4; i += blockDim.x) z[i] = make_uint4(0, 0, 0, 0);
}

/* ---- histogram of a share with one CTA per SM --------------------------- */
/* Counters: word 64 v + 32 c + lane counts bin v for one lane of copy c, in a
 * 64 KB table that starts on a 64 KB boundary of the shared window.  A bin's
 * row is 256 bytes, so byte 1 of a counter's address is the bin itself and
 * the other three bytes belong to the lane: one byte permute of the loaded
 * word and the lane's base makes each address (no add).  Lane l only touches
 * bank l.  The addresses are formed four reductions ahead.
 * What bounds it is the shared-memory pipe: 512 bytes of input cost 16 warp
 * reductions, a 128-bit read per lane (4 wavefronts) and the TMA write of the
 * same bytes (4), 24 clocks or 21.3 bytes a clock.  Measured per SM: 20.4 with
 * HBM idle (38 CTAs), 19 on 152 CTAs (3 x 1 GiB in one launch, boot included:
 * 5.7 TB/s; with a permute and an add per address, and two copies to clear and
 * read, 16.6 and 5.2).
 * Loads straight into registers instead of through the ring: 21.1 on 38 CTAs,
 * but 5.24 TB/s on 152, too few bytes in flight.  A second copy of the
 * counters only adds clearing and read-out. */
__device__ __forceinline__ uint32_t row_addr(uint32_t w, uint32_t lane_addr, uint32_t sel) {
  uint32_t r;
  asm volatile("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(w), "r"(lane_addr), "r"(sel));
  return r;
}
__device__ __forceinline__ void count16_row(uint32_t lane_addr, uint4 q) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
  uint32_t a[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) a[j] = row_addr(w[0], lane_addr, 0x7604u | ((uint32_t)j << 4));
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], 1;" ::"r"(a[j & 3]) : "memory");
    if (j < 12) a[j & 3] = row_addr(w[(j >> 2) + 1], lane_addr, 0x7604u | ((uint32_t)(j & 3) << 4));
  }
}

/* Shared-memory offset (from dsm) of the counter table; the rings lie around
 * it (lk_hist_ring_off). */
__device__ __forceinline__ uint32_t hist_table_off(const unsigned char* dsm) {
  return ((smem_addr(dsm) + 0xffffu) & ~0xffffu) - smem_addr(dsm);
}

/* Clear the counters of the copies in use (the first 128 * copies bytes of
 * each 256-byte row). */
template <uint32_t COPIES>
__device__ __forceinline__ void hist_row_zero(unsigned char* tbl) {
  constexpr uint32_t per_row = COPIES * 8u;   /* 16-byte words */
  for (uint32_t i = threadIdx.x; i < 256u * per_row; i += blockDim.x)
    *reinterpret_cast<uint4*>(tbl + (i / per_row) * 256u + (i % per_row) * 16u) = make_uint4(0, 0, 0, 0);
}

/* Thread v (< 256) adds row v (32 lanes of each copy); each 8-thread phase
 * of the 128-bit loads starts at thread-dependent columns and so touches all
 * 32 banks once. */
template <uint32_t COPIES>
__device__ __forceinline__ uint32_t hist_row_readout(const unsigned char* tbl, uint32_t v) {
  constexpr uint32_t per_row = COPIES * 8u;
  const uint4* rw = reinterpret_cast<const uint4*>(tbl + v * 256u);
  uint32_t tot = 0;
#pragma unroll
  for (uint32_t j = 0; j < per_row; ++j) {
    const uint4 q = rw[(j + v) & (per_row - 1u)];
    tot += (q.x + q.y) + (q.z + q.w);
  }
  return tot;
}

/* Every warp streams its own contiguous part of the CTA's share [beg, end)
 * (16-byte vectors) through a private ring of LK_STAGES stages (4 KB each at
 * 256 threads; six or eight smaller stages in the same memory were 10-25 %
 * slower, stages that are no multiple of 2 KB 11 %), which its
 * lane 0 fills with TMA bulk copies and all its lanes await on the warp's own
 * mbarriers (bars[LK_NUM_BARS + 4 w + s], phase bits LK_NUM_BARS + s of
 * `phase`, which every lane of the warp keeps alike).  A warp never waits for
 * another between chunks (with one ring per CTA, warps stalled about a fifth
 * of their cycles at the per-chunk barrier: random bytes make their counting
 * times uneven).  The first loads are issued before `before_count` runs on
 * the whole CTA (it clears the counters), so their latency covers it.
 * Returns false, on every thread alike, if a stage did not arrive before the
 * deadline. */
template <int P, bool PAIRS, bool YIELD, class F>
__device__ __forceinline__ bool hist_warp_streams(const uint4* in, uint64_t beg, uint64_t end, unsigned char* dsm,
                                                  uint64_t* bars, uint32_t& phase, uint32_t lane_addr, Pace pace,
                                                  F&& before_count) {
  static_assert(P == 1, "the counter rows need one CTA per SM's shared memory");
  const uint32_t W = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t stage_vec = lk_hist_stage_vecs(W);
  const uint32_t tbl = hist_table_off(dsm);
  const uint32_t ring_off = lk_hist_ring_off(W, warp, tbl);
  uint4* ring = reinterpret_cast<uint4*>(dsm + ring_off);
  uint64_t* wb = bars + LK_NUM_BARS + warp * LK_STAGES;
  uint64_t wbeg, wend;
  share(end - beg, (int)warp, (int)W, wbeg, wend);
  wbeg += beg;
  wend += beg;
  /* the warp's part, its ring slice and barriers, and the farthest counter
   * address any byte can form (row 255 of this lane and copy) */
  if (!LK_INB(wbeg <= wend && wend <= end, LK_OOB_SHARE) ||
      !LK_INB(tbl >= LK_HIST_QUARTER && ring_off + LK_STAGES * stage_vec * 16u <= LK_TC_SMEM &&
                  (smem_addr(ring) & 15u) == 0 &&
                  (ring_off >= tbl + LK_HIST_TABLE || ring_off + LK_STAGES * stage_vec * 16u <= tbl) &&
                  LK_NUM_BARS + (warp + 1) * LK_STAGES <= LK_ALL_BARS, LK_OOB_STREAM_SMEM) ||
      !LK_INB(((lane_addr >> 8) & 0xffu) == 0 && lane_addr - smem_addr(dsm) >= tbl &&
                  lane_addr - smem_addr(dsm) + 0xff00u + 4u <= tbl + LK_HIST_TABLE, LK_OOB_HIST_COUNTER))
    wend = wbeg;
  const uint64_t total = wend - wbeg;
  const uint64_t nch = (total + stage_vec - 1) / stage_vec;
  /* the warp's rate: the CTA's, split evenly over its warps */
  const uint64_t rate = pace.rate ? (pace.rate / W ? pace.rate / W : 1) : 0;
  const uint64_t deadline =
      (rate ? pace.deadline + total * 16u * 1000u / rate : pace.deadline) + (YIELD ? LK_YIELD_BUDGET_NS : 0u);
  const uint64_t t_first = rate && lane == 0 ? gtime() : 0;
  /* compiled apart from the plain loop: its state would cost the counting
   * loop registers */
  Yield yield(YIELD && lane == 0 && nch ? pace.gate : nullptr);
  auto parity = [&](uint64_t ch) {
    return ((phase >> (LK_NUM_BARS + (uint32_t)(ch % LK_STAGES))) & 1u) ^ ((uint32_t)(ch / LK_STAGES) & 1u);
  };
  auto issue = [&](uint64_t ch) {   /* lane 0 only */
    const uint32_t st = (uint32_t)(ch % LK_STAGES);
    const uint64_t v0 = wbeg + ch * stage_vec;
    const uint32_t nv = (uint32_t)((wend - v0) < stage_vec ? (wend - v0) : stage_vec);
    if (!LK_INB(v0 + nv <= wend && ((uintptr_t)(in + v0) & 15u) == 0, LK_OOB_STREAM_LOAD)) {
      mbar_expect_tx(&wb[st], 0u);   /* skipped: the phase completes with no bytes */
      return;
    }
    mbar_expect_tx(&wb[st], nv * 16u);
    bulk_g2s(ring + (size_t)st * stage_vec, in + v0, nv * 16u, &wb[st]);
  };
  if (lane == 0 && nch) {
    if (YIELD) yield.hold();
    fence_proxy_async_global();   /* earlier generic writes before these async reads */
    fence_proxy_async_smem();     /* earlier generic shared accesses before async writes */
    for (uint64_t ch = 0; ch < nch && ch < LK_STAGES; ++ch) issue(ch);
  }
  __syncwarp();
  bool failed = !before_count();
  auto refill = [&](uint64_t ch) {   /* every lane has read chunk ch: its stage takes chunk ch + LK_STAGES */
    __syncwarp();
    if (lane == 0 && ch + LK_STAGES < nch) {
      /* token bucket as deep as the ring: chunk k >= LK_STAGES no earlier
       * than t_first + (k - LK_STAGES + 1) chunks' worth of time */
      if (rate) sleep_until(t_first + (ch + 1) * (uint64_t)stage_vec * 16u * 1000u / rate);
      if (YIELD) yield.hold();
      fence_proxy_async_smem();
      issue(ch + LK_STAGES);
    }
  };
  auto arrived = [&](uint64_t ch) {   /* warp-uniform */
    return __all_sync(0xffffffffu, mbar_wait(&wb[ch % LK_STAGES], parity(ch), deadline));
  };
  uint64_t ch = 0;
  /* At most eight warps (stages of 4 KB and more): whole chunks, in pairs of 2
   * KB batches (four vectors a lane), the next batch loaded before the current
   * one's 64 reductions are issued (they are ordered asm, so loads placed
   * after them would wait for them), across the stage wait too (against
   * loading a batch, then counting it: 128 threads, 4.65 -> 5.35 TB/s over 3 x
   * 1 GiB; 256 threads, 8 x 256 MiB in 422 -> 409 us). */
  const uint64_t nfull = stage_vec % 256u == 0 ? total / stage_vec : 0;
  if (PAIRS && nfull && !failed) {   /* PAIRS: kernels of at most 256 threads, which have the registers */
    uint4 q0[4], q1[4];
    auto load4 = [&](uint4 (&q)[4], const uint4* s0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) q[i] = s0[lane + 32 * i];
    };
    auto count4 = [&](const uint4 (&q)[4]) {
#pragma unroll
      for (int i = 0; i < 4; ++i) count16_row(lane_addr, q[i]);
    };
    failed = !arrived(0);
    load4(q0, ring);   /* a failed wait's bytes are not counted */
    for (; ch < nfull && !failed; ++ch) {
      const uint4* s0 = ring + (size_t)(ch % LK_STAGES) * stage_vec;
      load4(q1, s0 + 128);
      count4(q0);
      for (uint32_t v = 256; v < stage_vec; v += 256) {
        load4(q0, s0 + v);
        count4(q1);
        load4(q1, s0 + v + 128);
        count4(q0);
      }
      if (ch + 1 < nfull) {
        if (!arrived(ch + 1)) {
          failed = true;
          refill(ch++);   /* as after a counted chunk: LK_STAGES chunks from ch on are issued */
          break;
        }
        load4(q0, ring + (size_t)((ch + 1) % LK_STAGES) * stage_vec);
      }
      count4(q1);
      refill(ch);
    }
  }
  for (; ch < nch && !failed; ++ch) {
    if (!arrived(ch)) {
      failed = true;
      break;
    }
    const uint64_t v0 = wbeg + ch * stage_vec;
    const uint32_t cnt = (uint32_t)((wend - v0) < stage_vec ? (wend - v0) : stage_vec);
    const uint4* s0 = ring + (size_t)(ch % LK_STAGES) * stage_vec;
    uint32_t v = lane;
    for (; v + 96 < cnt; v += 128) {
      uint4 q[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) q[i] = s0[v + 32 * i];
#pragma unroll
      for (int i = 0; i < 4; ++i) count16_row(lane_addr, q[i]);
    }
    for (; v < cnt; v += 32) count16_row(lane_addr, s0[v]);
    refill(ch);
  }
  /* a failed wait leaves the copies issued after it in flight: let them land */
  const uint64_t issued = failed ? (ch + LK_STAGES < nch ? ch + LK_STAGES : nch) : nch;
  if (lane == 0)
    for (uint64_t c2 = ch; failed && c2 < issued; ++c2)
      mbar_wait(&wb[c2 % LK_STAGES], parity(c2), deadline + 1000000000ull);
  /* each issued chunk completed one phase of its stage's barrier */
  for (uint32_t st = 0; st < LK_STAGES; ++st) {
    const uint64_t uses = issued > st ? (issued - st + LK_STAGES - 1) / LK_STAGES : 0;
    phase ^= (uint32_t)(uses & 1u) << (LK_NUM_BARS + st);
  }
  return !__syncthreads_or(failed);
}

/* A persistent CTA's place and its last descriptors, in shared memory (so
 * that they cost the bodies no registers). */
struct lk_cta {
  lk_slot taken[LK_BCAST_DEPTH];   /* descriptor k (0-based) in [k mod D]: the last D taken        */
  lk_dcluster* dc;                 /* its cluster's device state                                   */
  uint64_t* done;                  /* its host-visible completion word                             */
  const uint64_t* abort;           /* the host's abort word                                        */
  uint64_t patience;               /* wait_finished: limit without progress (ns), 0 = the body's   */
  int32_t cl, rank, size;          /* cluster (-1: none), rank in it, the cluster's CTAs           */
  uint64_t t_pick[2], t_start[2];  /* stamps of descriptor k in [k mod 2], for the execution log   */
  uint64_t t_end;                  /* when the last body ended                                     */
};

/* Where a histogram's counts go.  With both pointers null, this CTA counts all
 * of it and stores the bins.  With `acc` set, every CTA adds its counts into
 * it (zero at rest) and a combine copies it out afterwards (split parts,
 * ordinary launches).  With `cta` set (descriptor `seq` of a
 * cluster), rank 0 clears the output itself and release-stores seq into the
 * slot's clear word, and every CTA adds its counts straight into the output
 * once it has acquired that word: no combine, and no CTA waits for another at
 * the end.
 * Rank 0 clears only once every earlier descriptor of the cluster that
 * touches the output has finished on every CTA, so a CTA still writing or
 * reading the same buffer for an earlier descriptor cannot meet the clear:
 * the output ends as the last descriptor's result, as if the descriptors ran
 * one by one.  The ones that can still be running are the 7 before this one
 * (a slot is reused once its descriptor finished).  With outputs apart rank 0
 * does not wait: waiting for the previous descriptor, whatever it was, made
 * every histogram wait for the slowest CTA. */
struct HistSink {
  uint32_t* acc;
  const lk_cta* cta;
  uint64_t seq;
  __device__ __forceinline__ uint64_t* clear_word() const { return &cta->dc->hzero[(seq - 1) % LK_BCAST_DEPTH]; }
};

/* Does descriptor e read or write any byte of [lo, hi)?  (A batch or the
 * serving queue may.) */
__device__ __forceinline__ bool touches(const lk_slot& e, uint64_t lo, uint64_t hi) {
  uint64_t b0 = 0, b1 = 0, bo = 0;
  switch (e.cmd - LK_CMD_WORK) {
    case LK_OP_NOP: return false;
    case LK_OP_ADD_I32: b0 = b1 = bo = 4 * e.n; break;
    case LK_OP_COPY_I32: b0 = bo = 4 * e.n; break;
    case LK_OP_HIST_U8: b0 = e.n; bo = 1024; break;
    case LK_OP_SUM_F32: b0 = 4 * e.n; bo = 4; break;
    case LK_OP_GEMM64_F32: b0 = b1 = bo = 16384 * e.n; break;
    case LK_OP_COMBINE_SUM: b0 = 16 * e.n; bo = 4; break;
    case LK_OP_COMBINE_HIST: b0 = 1024 * e.n; bo = 1024; break;
    case LK_OP_SPIN: bo = 4 * LK_MAX_CTAS; break;
    default: return true;
  }
  return (e.in0 < hi && e.in0 + b0 > lo) || (e.in1 < hi && e.in1 + b1 > lo) || (e.out < hi && e.out + bo > lo);
}

/* One thread: wait until another CTA's word reaches `want`; false if it does
 * not in time.  The limit is the body's deadline, except in finite lists whose
 * CTAs read the ring themselves (`patience`): there this CTA may be up to eight
 * descriptors ahead of the one it waits for, whose bodies do not count against
 * this one, so the wait goes on while the cluster finishes descriptors. */
__device__ __noinline__ bool wait_finished(const lk_cta* cta, const uint64_t* word, uint64_t want, uint64_t deadline) {
  const uint64_t limit = cta->patience;
  lk_patience p = {0, limit ? gtime() + limit : deadline};
  for (uint32_t it = 1;; ++it) {
    if (ld_acquire_gpu(word) >= want) return true;
    if (it & 63u) continue;
    uint64_t progress = 0;
    if (limit) {
      if (ld_relaxed_sys(cta->abort) || ld_relaxed_gpu(&cta->dc->gen) == LK_GEN_STOP) return false;
      for (uint32_t i = 0; i < LK_BCAST_DEPTH; ++i) progress += ld_relaxed_gpu(&cta->dc->slot_done[i]);
    }
    if (lk_out_of_patience(&p, gtime(), progress, limit)) return false;
  }
}

/* Rank 0, the whole CTA: wait for the earlier descriptors that touch the
 * output of descriptor `seq` (one lane of warp 0 each); false, on every
 * thread, if one did not finish in time. */
__device__ __noinline__ bool hist_may_clear(const lk_cta* cta, uint64_t seq, uint64_t deadline) {
  __shared__ int s_clear;
  if (threadIdx.x < 32) {
    const uint64_t k = seq - 1, back = threadIdx.x + 1, out = cta->taken[k % LK_BCAST_DEPTH].out;
    bool ok = true;
    if (back < LK_BCAST_DEPTH && back <= k) {
      const uint32_t i = (uint32_t)((k - back) % LK_BCAST_DEPTH);
      if (touches(cta->taken[i], out, out + 1024))
        ok = wait_finished(cta, &cta->dc->slot_done[i], k - back + 1, deadline);
    }
    ok = __all_sync(0xffffffffu, ok);
    if (threadIdx.x == 0) s_clear = ok;
  }
  __syncthreads();
  return s_clear != 0;
}

/* Thread 0 waits for rank 0's cleared output (with a sink that has one),
 * then the whole CTA synchronises; false, on every thread, if the word did
 * not arrive in time. */
__device__ __forceinline__ bool hist_out_ready(const HistSink& sink, uint64_t deadline) {
  __shared__ int s_ready;
  if (threadIdx.x == 0)
    s_ready = !sink.cta || ld_acquire_gpu(sink.clear_word()) >= sink.seq ||
              wait_finished(sink.cta, sink.clear_word(), sink.seq, deadline);
  __syncthreads();
  return s_ready != 0;
}

template <int P, bool PAIRS>
__device__ __forceinline__ bool body_hist(const lk_slot& d, int r, int S, unsigned char* dsm, uint64_t* bars,
                                          uint32_t& phase, Pace pace, HistSink sink) {
  const uint64_t nv = d.n >> 4;
  uint64_t beg, end;
  share(nv, r, S, beg, end);
  if (!LK_INB(beg <= end && end <= nv, LK_OOB_SHARE)) end = beg;
  const bool tail = (r == S - 1) && (d.n & 15);
  const uint32_t T = blockDim.x, W = T / 32, lane = threadIdx.x & 31;
  uint32_t* sh = reinterpret_cast<uint32_t*>(dsm);
  const uint8_t* xb = reinterpret_cast<const uint8_t*>(d.in0);
  const uint4* in = reinterpret_cast<const uint4*>(d.in0);
  bool ok = true;
  const uint64_t total = end - beg;
  uint32_t* acc = sink.acc ? sink.acc : reinterpret_cast<uint32_t*>(d.out);
  const bool alone = !sink.acc && !sink.cta;
  /* rank 0 of a cluster: the counts' targets start at zero;
   * the others add once they see it */
  auto clear_out = [&]() -> bool {
    if (!sink.cta || r != 0) return true;
    if (!hist_may_clear(sink.cta, sink.seq, pace.deadline)) return false;
    for (uint32_t v = threadIdx.x; v < 256; v += T) acc[v] = 0;
    __syncthreads();
    if (threadIdx.x == 0) st_release_gpu(sink.clear_word(), sink.seq);
    return true;
  };
  if (total * 16 < LK_HIST_SMALL_BYTES) {
    if (!clear_out()) return false;
    hist_zero(sh, W * 256);
    __syncthreads();
    uint32_t* bins = sh + (threadIdx.x >> 5) * 256;
    ok = stream<1, false, P>(in, nullptr, beg, end, dsm + SmemCfg<P>::work_bytes, bars, phase,
                          pace, [&](uint64_t, uint32_t cnt, const uint4* s0, const uint4*) {
                            for (uint32_t v = threadIdx.x; v < cnt; v += T) {
                              const uint4 q = s0[v];
                              count4_warp(bins, q.x);
                              count4_warp(bins, q.y);
                              count4_warp(bins, q.z);
                              count4_warp(bins, q.w);
                            }
                          });
    if (tail)
      for (uint64_t j = nv * 16 + threadIdx.x; j < d.n; j += T) atomicAdd(&bins[xb[j]], 1u);
    const bool ready = hist_out_ready(sink, pace.deadline);
    for (uint32_t v = threadIdx.x; ready && v < 256; v += T) {
      uint32_t s = 0;
      for (uint32_t w = 0; w < W; ++w) s += sh[w * 256 + v];
      if (alone) acc[v] = s;
      else if (s) atomicAdd(&acc[v], s);
    }
    return ok && ready;
  }
  if constexpr (P == 1) {
    /* one CTA per SM: rows of lane-private counters, all warps of a copy
     * share its words (their reductions are atomic) */
    constexpr uint32_t copies = LK_HIST_COPIES;
    unsigned char* tbl = dsm + hist_table_off(dsm);
    const uint32_t lane_addr = smem_addr(tbl) + ((threadIdx.x >> 5) % copies) * 128u + lane * 4u;
    auto prepare = [&]() -> bool {
      hist_row_zero<copies>(tbl);
      const bool cleared = clear_out();
      __syncthreads();
      return cleared;
    };
    ok = pace.gate ? hist_warp_streams<P, false, true>(in, beg, end, dsm, bars, phase, lane_addr, pace, prepare)
                   : hist_warp_streams<P, PAIRS, false>(in, beg, end, dsm, bars, phase, lane_addr, pace, prepare);
    if (tail)
      for (uint64_t j = nv * 16 + threadIdx.x; j < d.n; j += T)
        asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], 1;" ::"r"(lane_addr + ((uint32_t)xb[j] << 8))
                     : "memory");
    const bool ready = hist_out_ready(sink, pace.deadline);
    for (uint32_t v = threadIdx.x; ready && v < 256; v += T) {
      const uint32_t tot = hist_row_readout<copies>(tbl, v);
      if (alone) acc[v] = tot;
      else if (tot) atomicAdd(&acc[v], tot);
    }
    return ok && ready;
  } else {
    /* two CTAs per SM: one ring for the CTA; lane-private 32-bit counters,
     * shared by the CTA's warps (their reductions to a word are atomic) */
    if (!clear_out()) return false;
    constexpr uint32_t copies = SmemCfg<P>::hist_copies;
    const uint32_t copy = (threadIdx.x >> 5) % copies;
    const uint32_t lane_addr = smem_addr(sh + copy * 8192u + lane);
    hist_zero(sh, copies * 8192u);
    __syncthreads();
    ok = stream<1, false, P>(in, nullptr, beg, end, dsm + SmemCfg<P>::work_bytes, bars, phase,
                          pace, [&](uint64_t, uint32_t cnt, const uint4* s0, const uint4*) {
                            /* four vectors loaded before their 64 reductions: the
                             * reductions are ordered asm, so loads placed after
                             * them would wait for them */
                            uint32_t v = threadIdx.x;
                            for (; v + 3 * T < cnt; v += 4 * T) {
                              uint4 q[4];
#pragma unroll
                              for (int i = 0; i < 4; ++i) q[i] = s0[v + i * T];
#pragma unroll
                              for (int i = 0; i < 4; ++i) {
                                count4_lane(lane_addr, q[i].x);
                                count4_lane(lane_addr, q[i].y);
                                count4_lane(lane_addr, q[i].z);
                                count4_lane(lane_addr, q[i].w);
                              }
                            }
                            for (; v < cnt; v += T) {
                              const uint4 q = s0[v];
                              count4_lane(lane_addr, q.x);
                              count4_lane(lane_addr, q.y);
                              count4_lane(lane_addr, q.z);
                              count4_lane(lane_addr, q.w);
                            }
                          });
    if (tail)
      for (uint64_t j = nv * 16 + threadIdx.x; j < d.n; j += T)
        asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], 1;" ::"r"(lane_addr + ((uint32_t)xb[j] << 7)) : "memory");
    const bool ready = hist_out_ready(sink, pace.deadline);
    for (uint32_t v = threadIdx.x; ready && v < 256; v += T) {
      const uint32_t tot = hist_readout<P>(sh, v);
      if (alone) acc[v] = tot;
      else if (tot) atomicAdd(&acc[v], tot);
    }
    return ok && ready;
  }
}

/* Threads t of `stride`: copy the accumulator out and return it to zero for reuse. */
__device__ __forceinline__ void combine_hist(const lk_slot& d, uint32_t* acc, uint32_t t, uint32_t stride) {
  int32_t* out = reinterpret_cast<int32_t*>(d.out);
  for (uint32_t v = t; v < 256; v += stride) {
    out[v] = (int32_t)__ldcg(acc + v);
    acc[v] = 0;
  }
}

/* ---- the compute-bound loop (Sec. III) ----------------------------------- */
__device__ __forceinline__ void body_spin(const lk_slot& d, int r, uint32_t* red) {
  uint32_t x = 65536u * (uint32_t)r + threadIdx.x + 1u;
  /* 32 dependent steps per trip: the 64-bit counter and the back edge cost some
   * ten clocks a trip (20k steps, eight per trip: 43 to 51 us, depending on the
   * code around the loop; 32: 45).  Each step is an instruction of its own: left to
   * the compiler, several are folded into one multiply-add. */
  const uint64_t n = d.n;
  uint64_t i = 0;
  auto step = [&]() { asm volatile("mad.lo.u32 %0, %0, %1, %2;" : "+r"(x) : "r"(1664525u), "r"(1013904223u)); };
#pragma unroll 1
  for (; i + 32 <= n; i += 32) {
#pragma unroll
    for (int j = 0; j < 32; ++j) step();
  }
#pragma unroll 1
  for (; i < n; ++i) step();
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x ^= __shfl_xor_sync(0xffffffffu, x, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x == 0 && d.out) {
    uint32_t v = 0;
    for (uint32_t w = 0; w < blockDim.x / 32; ++w) v ^= red[w];
    reinterpret_cast<uint32_t*>(d.out)[r] = v;
  }
}

/* ---- clearing (lk_serve's queue state) ------------------------------------ */
__device__ __forceinline__ void body_zero(const lk_slot& d, int r, int S) {
  uint64_t beg, end;
  share(d.n >> 4, r, S, beg, end);
  uint4* o = reinterpret_cast<uint4*>(d.out);
  for (uint64_t v = beg + threadIdx.x; v < end; v += blockDim.x)
    if (LK_INB(v < d.n >> 4, LK_OOB_STORE)) o[v] = make_uint4(0, 0, 0, 0);
}

/* ---- combining chunk results (rank 0 of the cluster alone) ------------- */
/* out[0] = binary64 sum of n float32 partials, one per 16-byte slot, added
 * lane-strided then by a fixed shuffle tree: the order depends only on n. */
__device__ __forceinline__ void body_combine_sum(const lk_slot& d, int r) {
  if (r != 0 || threadIdx.x >= 32) return;
  const float* p = reinterpret_cast<const float*>(d.in0);
  double s = 0.0;
  for (uint64_t q = threadIdx.x; q < d.n; q += 32) s += (double)__ldcg(p + 4 * q);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (threadIdx.x == 0) *reinterpret_cast<float*>(d.out) = (float)s;
}

/* out[v] = sum over j < n of in0[256 j + v]: n int32 histograms. */
__device__ __forceinline__ void body_combine_hist(const lk_slot& d, int r) {
  if (r != 0) return;
  const int32_t* h = reinterpret_cast<const int32_t*>(d.in0);
  for (uint32_t v = threadIdx.x; v < 256; v += blockDim.x) {
    uint32_t s = 0;
    for (uint64_t j = 0; j < d.n; ++j) s += (uint32_t)__ldcg(h + 256 * j + v);
    reinterpret_cast<int32_t*>(d.out)[v] = (int32_t)s;
  }
}

/* ---- 64x64x64 float32 GEMM tiles ---------------------------------------- */
/* Work unit = (tile, block of 64/U rows).  U > 1 only when there are fewer
 * tiles than CTAs, so that one tile can spread over up to 8 CTAs. */
__device__ __forceinline__ uint32_t gemm_row_split(uint64_t tiles, int S) {
  uint32_t U = 1;
  if (tiles > 0 && tiles < (uint64_t)S) {
    uint64_t want = ((uint64_t)S + tiles - 1) / tiles;
    while (U < want && U < 8) U <<= 1;
  }
  return U;
}

/* Shared memory: SmemCfg<P>::gemm_stages stages of (A rows 16 KB, B tile
 * 16 KB) over the whole dynamic shared memory; one mbarrier per stage. */

/* ---- the GEMM tile on the 5th-generation tensor cores ------------------- */
/* C = A B for whole 64x64x64 float32 tiles, with tcgen05.mma kind::f16 on
 * bf16 operands (exact products, float32 accumulation in TMEM).  One bf16
 * (or TF32) product per element pair would miss the 1e-4 sum|a b| bound, so
 * every operand is split in two: x_hi = bf16(x) and x_lo = bf16(x - x_hi),
 * both rounded to nearest; x - x_hi is exact in float32, and x_hi + x_lo
 * differs from x by at most 2^-16 |x|, so each product a b is formed to
 * within about 2^-15 |a b| (3.1e-5, against the 1e-4 bound).  What the tensor
 * core's accumulation adds is not specified; measured against binary64 the
 * whole error is at most 3.9e-6 sum |a b| (2,048 tiles of N(0,1)).  A_lo and A_hi accumulate along K and
 * B_hi and B_lo lie side by side along N, so eight MMAs (M = 64, N = 128,
 * K = 16) leave all four products of a tile in a 64 x 128 TMEM block, and
 * C[r][n] = D[r][n] + D[r][n + 64]: one thread holds both, nothing is
 * exchanged between threads.  A is K-major and B MN-major (its rows lie along
 * N in memory), so both operands are split the same way, row by row, with no
 * transposition: 64 bf16 are the 128 bytes of one swizzled row.
 *
 * The CTA's eight warps split tile k into operand buffer k mod 2, one thread
 * hands it to the tensor core and refills the raw stage, and while those MMAs
 * run every warp stores its part of tile k-1: one barrier per tile.
 * What bounds it is HBM: 3 x 2^15 tiles move 6.57 TB/s once booted (6.5 with
 * the boot), as much as
 * the same loads and stores with neither split nor MMAs (6.63).  One SM alone
 * (38 CTAs, HBM idle) takes 2,060 clocks a tile, against 2,275 of its share of
 * HBM: 1,130 for the loads and stores, the rest for the split and the chain
 * through the MMAs, which take 512 clocks themselves.  Operands stacked along
 * M and N instead (four MMAs of 128 x 128), B transposed on the way and the
 * column and row halves added through shared memory moved 5.95 TB/s.  A fifth
 * stage gains nothing.
 * Shared memory: four 32 KB TMA stages of raw tiles (A, then B) at 0; two
 * 32 KB operand buffers (A_hi, A_lo, B_hi, B_lo) from the next 1 KB boundary.
 * TMEM: 256 columns (two blocks of 128), allocated for the body and freed on
 * every path out of it. */
#define LK_TC_STAGES 4u
#define LK_TC_MMA_BAR 4u            /* bars 4, 5: MMA completion of operand buffer b */
#define LK_TC_OPS (128u * 1024u)    /* at least: rounded up to 1 KB of the shared window */
#define LK_TC_COLS 256u
/* instruction descriptor: D float32 (bits 4-5 = 1), A and B bf16 (bits 7-9,
 * 10-12 = 1), A K-major, B MN-major (bit 16), N = 128 (bits 17-22 = N/8),
 * M = 64 (bits 24-28 = M/16) */
#define LK_TC_IDESC ((1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((128u >> 3) << 17) | ((64u >> 4) << 24))

/* (x0, x1) -> bf16 pairs hi = bf16(x), lo = bf16(x - hi), x0 in the low half */
__device__ __forceinline__ void bf16_split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(x1), "f"(x0));
  const float h0 = __uint_as_float(hi << 16), h1 = __uint_as_float(hi & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(x1 - h1), "f"(x0 - h0));
}

/* The 256 threads: split the staged raw tile (A rows at `raw`, B rows at
 * raw + 16 KB) into an operand buffer (hi rows of A, lo rows of A, hi of B, lo
 * of B, 8 KB each).  Row i of 64 bf16 takes 128 bytes at i 128, its 16-byte
 * chunk c at position c ^ (i % 8) (the 128-byte swizzle).  Warp w takes rows
 * 8 w .. 8 w + 7 of each operand; lane l takes 4-element quarters l % 8 and
 * l % 8 + 8 of two rows.  An 8-lane phase of the 128-bit reads covers 128
 * contiguous bytes; the 16 lanes of a 64-bit write cover half a row of two
 * rows whose numbers differ in bit 2, so in distinct banks. */
__device__ __forceinline__ void tc_split(const unsigned char* raw, unsigned char* ops, uint32_t t) {
  const uint32_t w = t >> 5, q = t & 7u, sl = (t >> 3) & 3u;
  const uint32_t r0 = (sl & 1u) * 4u + (sl >> 1);          /* then r0 + 2 */
  const unsigned char* src = raw + (8u * w + r0) * 256u + q * 16u;
  float4 x[8];
#pragma unroll
  for (uint32_t i = 0; i < 8; ++i)                         /* operand i / 4, row r0 + 2 (i / 2 % 2), half i % 2 */
    x[i] = *reinterpret_cast<const float4*>(src + (i >> 2) * 16384u + ((i >> 1) & 1u) * 512u + (i & 1u) * 128u);
  const uint32_t dst0 = (8u * w + r0) * 128u + (((q >> 1) ^ r0) << 4) + (q & 1u) * 8u;
#pragma unroll
  for (uint32_t i = 0; i < 8; ++i) {
    /* row + 2: 256 bytes on, chunk position ^ 2; second half: position ^ 4 */
    unsigned char* dst = ops + (i >> 2) * 16384u + ((dst0 ^ ((((i >> 1) & 1u) << 5) | ((i & 1u) << 6))) + ((i >> 1) & 1u) * 256u);
    uint2 hi, lo;
    bf16_split2(x[i].x, x[i].y, hi.x, lo.x);
    bf16_split2(x[i].z, x[i].w, hi.y, lo.y);
    *reinterpret_cast<uint2*>(dst) = hi;
    *reinterpret_cast<uint2*>(dst + 8192u) = lo;
  }
}

__device__ __forceinline__ bool body_gemm_tc(const lk_slot& d, int r, int S, unsigned char* dsm, uint64_t* bars,
                                             uint32_t& phase, Pace pace) {
  uint64_t beg, end;
  share(d.n, r, S, beg, end);
  if (!LK_INB(end <= d.n, LK_OOB_SHARE)) end = beg;
  if (beg >= end) return true;
  const float* A = reinterpret_cast<const float*>(d.in0) + beg * 4096;
  const float* B = reinterpret_cast<const float*>(d.in1) + beg * 4096;
  float* C = reinterpret_cast<float*>(d.out) + beg * 4096;
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  const uint32_t uwarp = __shfl_sync(0xffffffffu, warp, 0);   /* the same, known to be warp-uniform */
  const uint32_t tiles = (uint32_t)(end - beg);   /* at most 2^28 */
  constexpr uint64_t unit_bytes = 32768u;
  const uint64_t deadline = pace.rate ? pace.deadline + tiles * unit_bytes * 1000u / pace.rate : pace.deadline;
  const uint64_t t_first = pace.rate ? gtime() : 0;
  auto issue = [&](uint32_t u) {   /* one thread: tile u of the share into its stage */
    const uint32_t st = u % LK_TC_STAGES;
    unsigned char* sa = dsm + st * 32768u;
    fence_proxy_async_smem();
    if (!LK_INB(u < tiles, LK_OOB_GEMM_LOAD) || !LK_INB((st + 1) * 32768u <= LK_TC_OPS, LK_OOB_GEMM_SMEM)) {
      mbar_expect_tx(&bars[st], 0u);   /* skipped: the phase completes with no bytes */
      return;
    }
    mbar_expect_tx(&bars[st], 32768u);
    bulk_g2s(sa, A + (uint64_t)u * 4096, 16384u, &bars[st]);
    bulk_g2s(sa + 16384u, B + (uint64_t)u * 4096, 16384u, &bars[st]);
  };
  /* parity of a barrier's k-th completion in this body, from its bit at entry */
  auto parity = [&](uint32_t bar, uint32_t k) { return ((phase >> bar) & 1u) ^ (k & 1u); };
  __shared__ uint32_t s_tmem;
  __syncthreads();          /* every stage is free: the previous use ended with a barrier */
  if (threadIdx.x == 0) {
    fence_proxy_async_global();   /* earlier generic writes before these async reads */
    for (uint32_t u = 0; u < tiles && u < LK_TC_STAGES; ++u) issue(u);
  }
  if (warp == 0) {
    __syncwarp();
    tmem_alloc(&s_tmem, LK_TC_COLS);
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = s_tmem;
  /* both operand buffers inside the shared memory, both blocks in the allocated columns */
  unsigned char* ops0 = dsm + (((smem_addr(dsm) + LK_TC_OPS + 1023u) & ~1023u) - smem_addr(dsm));
  const bool bufs_ok =
      LK_INB((uint32_t)(ops0 - dsm) >= LK_TC_STAGES * 32768u && (uint32_t)(ops0 - dsm) + 2u * 32768u <= LK_TC_SMEM &&
                 (smem_addr(ops0) & 1023u) == 0 && 2u * 128u <= LK_TC_COLS,
             LK_OOB_GEMM_SMEM);
  /* M = 64: row m of the block is TMEM lane 32 (m / 16) + m % 16, so warp w
   * reads rows 16 (w % 4) .. + 15, columns 32 (w / 4) .. + 31 of both halves
   * (warps w and w + 4 share a quarter of the lanes).  Of every 8 columns a lane holds
   * two neighbours in rows lane / 4 and lane / 4 + 8: four lanes write one
   * 32-byte sector. */
  const uint32_t crow = 16u * (warp & 3u) + (lane >> 2), ccol = 32u * (warp >> 2) + 2u * (lane & 3u);
  const uint32_t dt = tmem + ((32u * (warp & 3u)) << 16) + 32u * (warp >> 2);
  /* Tile u from buffer u & 1: wait for its MMAs, then TMEM -> registers ->
   * global memory.  False if the MMAs did not complete in time. */
  auto epilogue = [&](uint32_t u) -> bool {
    const uint32_t b = u & 1u;
    if (!mbar_wait(&bars[LK_TC_MMA_BAR + b], parity(LK_TC_MMA_BAR + b, u >> 1), deadline + 1000000000ull)) return false;
    __syncwarp();
    tc_fence_after_sync();
    float v[16], w[16];
    tmem_ld_16x256b_x4_2(dt + 128u * b, dt + 128u * b + 64u, v, w);
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] += w[i];
    float* c = C + (uint64_t)u * 4096 + crow * 64u + ccol;
    if (LK_INB(u < tiles && crow + 8u < 64u && ccol + 26u <= 64u, LK_OOB_GEMM_STORE)) {
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        st_stream(reinterpret_cast<float2*>(c + 8u * j), make_float2(v[4 * j], v[4 * j + 1]));
        st_stream(reinterpret_cast<float2*>(c + 8u * j + 512u), make_float2(v[4 * j + 2], v[4 * j + 3]));
      }
    }
    return true;
  };
  bool ok = true;           /* this thread's waits; agreed at each barrier */
  uint32_t k = 0;           /* tiles handed to the tensor core */
  for (; k < tiles; ++k) {
    const uint32_t st = k % LK_TC_STAGES, b = k & 1u;
    unsigned char* ops = ops0 + 32768u * b;
    if (ok) ok = mbar_wait(&bars[st], parity(st, k / LK_TC_STAGES), deadline);
    if (ok) tc_split(dsm + st * 32768u, ops, threadIdx.x);   /* the buffer's last MMAs (tile k-2) have been waited for */
    fence_proxy_async_smem();       /* the operands, written by threads, are read by the tensor core */
    tc_fence_before_sync();         /* the TMEM reads of tile k-2 precede this block's next MMAs */
    if (!__syncthreads_and(ok)) {
      ok = false;
      break;
    }
    if (uwarp == 0) {
      if (elect_one()) {
        tc_fence_after_sync();
        if (bufs_ok) {
          const uint32_t base = smem_addr(ops);
#pragma unroll
          for (uint32_t p = 0; p < 2; ++p)                       /* A_lo, then A_hi */
#pragma unroll
            for (uint32_t j = 0; j < 4; ++j)                     /* K = 16 each */
              umma_f16(tmem + 128u * b, umma_desc_sw128(base + (1u - p) * 8192u + 32u * j, 16u, 1024u),
                       umma_desc_sw128(base + 16384u + 2048u * j, 8192u, 1024u), LK_TC_IDESC, (p | j) != 0);
        }
        umma_commit(&bars[LK_TC_MMA_BAR + b]);
      }
      __syncwarp();
    } else if (threadIdx.x == 32 && k + LK_TC_STAGES < tiles) {
      /* every thread has split tile k: its stage takes tile k + 4 */
      if (pace.rate) sleep_until(t_first + (k + 1) * unit_bytes * 1000u / pace.rate);
      issue(k + LK_TC_STAGES);
    }
    /* while the tensor core works on tile k, finish the previous tile */
    if (k > 0) ok = epilogue(k - 1);
  }
  if (ok) ok = epilogue(tiles - 1);
  ok = __syncthreads_and(ok);
  if (!ok && threadIdx.x == 0) {
    /* copies and MMAs may still be in flight: let them end (bounded) before
     * the stages and TMEM are given back; the last commit covers every MMA */
    for (uint32_t u = k; u < tiles && u < k + LK_TC_STAGES; ++u)
      mbar_wait(&bars[u % LK_TC_STAGES], parity(u % LK_TC_STAGES, u / LK_TC_STAGES), deadline + 1000000000ull);
    if (k > 0) {
      const uint32_t bar = LK_TC_MMA_BAR + ((k - 1) & 1u);
      mbar_wait(&bars[bar], parity(bar, (k - 1) >> 1), deadline + 2000000000ull);
    }
  }
  tc_fence_before_sync();
  __syncthreads();          /* stages, operand buffers and TMEM are free */
  tc_fence_after_sync();
  if (warp == 0) tmem_dealloc(tmem, LK_TC_COLS);
  /* every thread advances every barrier's phase bit by its completions here */
  if (ok) {
    for (uint32_t sb = 0; sb < LK_TC_STAGES; ++sb) {
      const uint32_t uses = tiles > sb ? (tiles - sb + LK_TC_STAGES - 1) / LK_TC_STAGES : 0;
      phase ^= (uses & 1u) << sb;
    }
    for (uint32_t b = 0; b < 2; ++b) {
      const uint32_t commits = tiles > b ? (tiles - b + 1) / 2 : 0;
      phase ^= (commits & 1u) << (LK_TC_MMA_BAR + b);
    }
  }
  return ok;
}

/* FFMA micro-tiles of one row block: `rows` rows of A (row-major, 64 k
 * each) times the 64 x 64 B tile, both in shared memory, into C (row-major,
 * 64 floats a row).  Thread t takes micro-tiles of MR rows x MC columns, t
 * and t + T ...; every output accumulates its 64 products in k order with
 * one fused multiply-add each, whatever the micro-tile shape, so a tile's
 * result does not depend on how it was split into row blocks. */
template <int MR, int MC, bool FULL_UNROLL>
__device__ __forceinline__ void ffma_block(const float* sA, const float* sB, float* cblk, uint32_t rows, bool store_ok) {
  constexpr uint32_t ncg = 64u / MC;
  const uint32_t nmt = rows / MR * ncg;
  for (uint32_t mt = threadIdx.x; mt < nmt; mt += blockDim.x) {
    const uint32_t r0 = mt / ncg * MR, c0 = mt % ncg * MC;
    float c[MR][MC];
#pragma unroll
    for (int i = 0; i < MR; ++i)
#pragma unroll
      for (int j = 0; j < MC; ++j) c[i][j] = 0.f;
#pragma unroll(FULL_UNROLL ? 16 : 2)
    for (uint32_t k = 0; k < 64; k += 4) {
      float av[MR][4], bv[4][MC];
#pragma unroll
      for (int i = 0; i < MR; ++i) {
        const float4 q = *reinterpret_cast<const float4*>(sA + (r0 + i) * 64 + k);
        av[i][0] = q.x; av[i][1] = q.y; av[i][2] = q.z; av[i][3] = q.w;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (MC == 4) {
          const float4 b = *reinterpret_cast<const float4*>(sB + (k + q) * 64 + c0);
          bv[q][0] = b.x; bv[q][1] = b.y; bv[q][MC > 2 ? 2 : 0] = b.z; bv[q][MC > 3 ? 3 : 0] = b.w;
        } else {
          const float2 b = *reinterpret_cast<const float2*>(sB + (k + q) * 64 + c0);
          bv[q][0] = b.x; bv[q][1] = b.y;
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < MR; ++i)
#pragma unroll
          for (int j = 0; j < MC; ++j) c[i][j] = fmaf(av[i][q], bv[q][j], c[i][j]);
    }
    if (store_ok && LK_INB(r0 + MR <= rows && c0 + MC <= 64u, LK_OOB_GEMM_STORE)) {
#pragma unroll
      for (int i = 0; i < MR; ++i) {
        float* crow = cblk + (r0 + i) * 64 + c0;
        if (MC == 4) *reinterpret_cast<float4*>(crow) = make_float4(c[i][0], c[i][1], c[i][MC > 2 ? 2 : 0], c[i][MC > 3 ? 3 : 0]);
        else *reinterpret_cast<float2*>(crow) = make_float2(c[i][0], c[i][1]);
      }
    }
  }
}

/* Whole tiles on the FFMA path, 256 threads: G groups of NT threads each take
 * every G-th tile of the share [beg, end), so while one group waits at the end
 * of its tile or for the next the others compute.  A thread accumulates 8 rows
 * x MC columns in packed float32 pairs (fma.rn.f32x2: two outputs a
 * multiply-add, each rounded as by fmaf), so every output is still its 64
 * products in k order.  Lane l of a warp takes column chunk l % 8 (and + 8 if
 * MC = 8) and rows 8 (l / 8) ..: an 8-lane phase of a 128-bit read covers 128
 * contiguous bytes of B, or one broadcast word of A.
 * What bounds it is the shared-memory pipe: 2,130 wavefronts of reads a tile
 * and 256 of the TMA's writes, 2,386 clocks, before the tile's 48 KB of an SM's
 * share of HBM (2,275) and the FP32 pipe (2,048).  Measured 2,940 clocks, 2 x
 * 32,768 tiles on 152 CTAs in 637 us (5.05 TB/s).  With 4 x 4 outputs a thread,
 * scalar fmaf and the whole CTA on one tile it was 4,480 and 950 us: twice the
 * shared-memory reads and instructions an output, and a CTA barrier a tile.
 * Two CTAs per SM (128 registers): 3.75 -> 3.96 TB/s.  A share of one tile is
 * left to the whole CTA (below), where one group alone would work on it: 24
 * descriptors of one tile a CTA in 132 us instead of 159; of two tiles the
 * groups take 171 and the whole CTA 182.
 * Stages are shared by the groups: tile u sits in stage (u - beg) % NST, and
 * the group that used it refills it; s_issued counts the loads issued into a
 * stage, since a parity wait is only sound one phase ahead. */
__device__ __forceinline__ uint64_t pack2(float a) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ void fma2(uint64_t& c, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
template <int P>
__device__ __forceinline__ bool body_gemm_ffma_tiles(const lk_slot& d, uint64_t beg, uint64_t end, unsigned char* dsm,
                                                     uint64_t* bars, uint32_t& phase, Pace pace) {
  constexpr uint32_t G = P == 1 ? 4 : 2, NT = 256 / G, MC = P == 1 ? 8 : 4, NP = MC / 2;
  constexpr int KU = P == 1 ? 4 : 1;   /* k chunks of 4 per loop trip (P = 1: 1, 2, 4, 16 gave 4.2, 4.8, 5.1, 4.5 TB/s) */
  constexpr uint32_t NST = P == 1 ? LK_TC_SMEM / 32768u : SmemCfg<P>::gemm_stages;   /* 7 or 3 */
  static_assert(NST <= LK_NUM_BARS && NST >= G, "one mbarrier per stage, a stage per group");
  const float* A = reinterpret_cast<const float*>(d.in0) + beg * 4096;
  const float* B = reinterpret_cast<const float*>(d.in1) + beg * 4096;
  float* C = reinterpret_cast<float*>(d.out) + beg * 4096;
  const uint32_t tiles = (uint32_t)(end - beg);
  const uint32_t g = threadIdx.x / NT, lt = threadIdx.x % NT, gw = lt >> 5, lane = threadIdx.x & 31u;
  /* P = 1: warp 0, 1 of a group take row groups 0-3, 4-7, all columns; P = 2: warps 2 i + j take row
   * groups 4 i .. and column half j */
  const uint32_t rg = (lane >> 3) + 4u * (MC == 8 ? gw : gw >> 1);
  const uint32_t col = 4u * (lane & 7u) + (MC == 8 ? 0u : 32u * (gw & 1u));
  constexpr uint64_t unit_bytes = 32768u;
  const uint64_t deadline = pace.rate ? pace.deadline + tiles * unit_bytes * 1000u / pace.rate : pace.deadline;
  const uint64_t t_first = pace.rate ? gtime() : 0;
  __shared__ uint32_t s_issued[NST];
  auto issue = [&](uint32_t u) {   /* one thread */
    const uint32_t st = u % NST;
    unsigned char* sa = dsm + st * 32768u;
    fence_proxy_async_smem();
    if (!LK_INB(u < tiles, LK_OOB_GEMM_LOAD) ||
        !LK_INB((st + 1) * 32768u <= (P == 1 ? LK_TC_SMEM : SmemCfg<P>::dyn_bytes), LK_OOB_GEMM_SMEM)) {
      mbar_expect_tx(&bars[st], 0u);   /* skipped: the phase completes with no bytes */
      return;
    }
    mbar_expect_tx(&bars[st], 32768u);
    bulk_g2s(sa, A + (uint64_t)u * 4096, 16384u, &bars[st]);
    bulk_g2s(sa + 16384u, B + (uint64_t)u * 4096, 16384u, &bars[st]);
  };
  auto parity = [&](uint32_t st, uint32_t use) { return ((phase >> st) & 1u) ^ (use & 1u); };
  __syncthreads();          /* every stage is free: the previous use ended with a barrier */
  if (threadIdx.x == 0) {
    fence_proxy_async_global();   /* earlier generic writes before these async reads */
    for (uint32_t st = 0; st < NST; ++st) {
      if (st < tiles) issue(st);
      s_issued[st] = st < tiles;
    }
  }
  __syncthreads();
  bool ok = true;
  for (uint32_t u = g; u < tiles; u += G) {
    const uint32_t st = u % NST, use = u / NST;
    const volatile uint32_t* iss = s_issued;
    for (uint32_t it = 0; ok && iss[st] < use + 1; ++it)
      if ((it & 15) == 15 && gtime() > deadline) ok = false;
    if (ok) ok = mbar_wait(&bars[st], parity(st, use), deadline);
    const float* sA = reinterpret_cast<const float*>(dsm + st * 32768u) + rg * 512u;
    const float* sB = reinterpret_cast<const float*>(dsm + st * 32768u + 16384u) + col;
    uint64_t c[8][NP];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < (int)NP; ++j) c[i][j] = 0;
    if (ok) {
#pragma unroll(KU)
      for (uint32_t k = 0; k < 64; k += 4) {
        float4 a[8];
        ulonglong2 b[4][NP / 2];
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = *reinterpret_cast<const float4*>(sA + i * 64 + k);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int h = 0; h < (int)NP / 2; ++h)
            b[q][h] = *reinterpret_cast<const ulonglong2*>(sB + (k + q) * 64 + 32 * h);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint64_t aa = pack2(q == 0 ? a[i].x : q == 1 ? a[i].y : q == 2 ? a[i].z : a[i].w);
#pragma unroll
            for (int h = 0; h < (int)NP / 2; ++h) {
              fma2(c[i][2 * h], aa, b[q][h].x);
              fma2(c[i][2 * h + 1], aa, b[q][h].y);
            }
          }
      }
    }
    /* the group has read the stage (and agrees whether it arrived) */
    if (!bar_sync_and(3u + g, NT, ok)) {
      ok = false;
      break;
    }
    if (lt == 0 && u + NST < tiles) {
      if (pace.rate) sleep_until(t_first + (u + 1) * unit_bytes * 1000u / pace.rate);
      issue(u + NST);
      __threadfence_block();
      atomicAdd(&s_issued[st], 1u);
    }
    float* ct = C + (uint64_t)u * 4096 + rg * 512u + col;
    if (LK_INB(u < tiles && rg * 8u + 8u <= 64u && col + 4u + 32u * (NP / 2 - 1) <= 64u, LK_OOB_GEMM_STORE)) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int h = 0; h < (int)NP / 2; ++h)
          *reinterpret_cast<ulonglong2*>(ct + i * 64 + 32 * h) = make_ulonglong2(c[i][2 * h], c[i][2 * h + 1]);
    }
  }
  ok = __syncthreads_and(ok);
  if (!ok) {
    /* copies may still be in flight: let every issued one land (bounded) */
    if (threadIdx.x == 0)
      for (uint32_t st = 0; st < NST; ++st)
        if (s_issued[st]) mbar_wait(&bars[st], parity(st, s_issued[st] - 1), deadline + 1000000000ull);
    __syncthreads();
    return false;
  }
#pragma unroll
  for (uint32_t st = 0; st < NST; ++st) {
    const uint32_t uses = tiles > st ? (tiles - st + NST - 1) / NST : 0;
    phase ^= (uses & 1u) << st;
  }
  return true;
}

/* Returns false if a staging copy did not complete before the deadline.
 * `phase` holds one parity bit per stage and persists across descriptors;
 * `pace` paces the tile loads as in stream().  Whole tiles at 256 threads
 * with one CTA per SM run on the tensor cores (body_gemm_tc) unless
 * `tensor_cores` is false; row blocks of split tiles and other shapes take
 * the FFMA path below. */
template <bool FULL_UNROLL, int P>
__device__ __forceinline__ bool body_gemm(const lk_slot& d, int r, int S, float* sm, uint64_t* bars,
                                          uint32_t& phase, Pace pace, bool tensor_cores) {
  const uint64_t tiles = d.n;
  const uint32_t U = gemm_row_split(tiles, S);
  /* FULL_UNROLL holds only in the kernels built for 256 threads and one CTA
   * per SM, the only ones that can take the tensor-core path */
  if constexpr (FULL_UNROLL)
    if (P == 1 && tensor_cores && U == 1 && blockDim.x == 256)
      return body_gemm_tc(d, r, S, reinterpret_cast<unsigned char*>(sm), bars, phase, pace);
  const uint32_t rows = 64 / U;
  uint64_t beg, end;
  share(tiles * U, r, S, beg, end);
  if (!LK_INB(end <= tiles * U, LK_OOB_SHARE)) end = beg;
  if (beg >= end) return true;
  if constexpr (FULL_UNROLL || P == 2)   /* the kernels of at most 256 threads */
    if (U == 1 && blockDim.x == 256 && end - beg > 1)
      return body_gemm_ffma_tiles<P>(d, beg, end, reinterpret_cast<unsigned char*>(sm), bars, phase, pace);
  const float* A = reinterpret_cast<const float*>(d.in0);
  const float* B = reinterpret_cast<const float*>(d.in1);
  float* C = reinterpret_cast<float*>(d.out);
  constexpr uint32_t nstages = SmemCfg<P>::gemm_stages;
  const uint64_t unit_bytes = rows * 256u + 16384u;
  const uint64_t deadline = pace.rate ? pace.deadline + (end - beg) * unit_bytes * 1000u / pace.rate : pace.deadline;
  const uint64_t t_first = pace.rate && threadIdx.x == 0 ? gtime() : 0;
  auto issue = [&](uint64_t u) {   /* thread 0 */
    const uint32_t st = (uint32_t)((u - beg) % nstages);
    const uint64_t tile = u / U;
    const uint32_t rb = (uint32_t)(u % U);
    float* sA = sm + st * LK_GEMM_STAGE_FLOATS;
    fence_proxy_async_smem();
    if (!LK_INB(tile < tiles && rb < U && (uint64_t)(rb + 1) * rows <= 64u, LK_OOB_GEMM_LOAD) ||
        !LK_INB((st + 1) * LK_GEMM_STAGE_FLOATS * 4u <= SmemCfg<P>::dyn_bytes, LK_OOB_GEMM_SMEM)) {
      mbar_expect_tx(&bars[st], 0u);   /* skipped: the phase completes with no bytes */
      return;
    }
    mbar_expect_tx(&bars[st], rows * 256u + 16384u);
    bulk_g2s(sA, A + tile * 4096 + (uint64_t)rb * rows * 64, rows * 256u, &bars[st]);
    bulk_g2s(sA + 4096, B + tile * 4096, 16384u, &bars[st]);
  };
  __shared__ int s_staged;
  __syncthreads();          /* every stage is free: the previous use ended with a barrier */
  if (threadIdx.x == 0) {
    fence_proxy_async_global();   /* earlier generic writes before these async reads */
    for (uint64_t u = beg; u < end && u < beg + nstages; ++u) issue(u);
  }
  bool ok = true;
  for (uint64_t u = beg; u < end; ++u) {
    const uint32_t st = (uint32_t)((u - beg) % nstages);
    /* thread 0 alone decides whether the stage arrived in time, so that every
     * thread takes the same path through the barriers below */
    if (threadIdx.x == 0) {
      int arrived = mbar_wait(&bars[st], (phase >> st) & 1u, deadline);
      if (!arrived) {
        /* let this CTA's own copies land before giving up */
        for (uint64_t v = u; v < end && v < u + nstages; ++v) {
          const uint32_t s2 = (uint32_t)((v - beg) % nstages);
          mbar_wait(&bars[s2], (phase >> s2) & 1u, deadline + 1000000000ull);
        }
      }
      s_staged = arrived;
    }
    __syncthreads();
    if (!s_staged) {
      ok = false;
      break;
    }
    /* every thread finished unit u-1: refill its stage with unit u-1+STAGES */
    if (threadIdx.x == 0 && u > beg && u - 1 + nstages < end) {
      if (pace.rate) sleep_until(t_first + (u - beg) * unit_bytes * 1000u / pace.rate);
      issue(u - 1 + nstages);
    }
    /* the phase is complete: this wait returns at once and makes the copied
     * bytes visible to this thread */
    mbar_wait(&bars[st], (phase >> st) & 1u, deadline + 1000000000ull);
    phase ^= 1u << st;
    const float* sA = sm + st * LK_GEMM_STAGE_FLOATS;
    const float* sB = sA + 4096;
    const uint64_t tile = u / U;
    const uint32_t rb = (uint32_t)(u % U);
    float* cblk = C + tile * 4096 + (uint64_t)rb * rows * 64;
    const bool cblk_ok = LK_INB(tile < tiles && (uint64_t)(rb + 1) * rows <= 64u, LK_OOB_GEMM_STORE);
    /* every thread takes a micro-tile: the smaller the row block, the fewer
     * outputs each (a one-tile item split 8 ways keeps all threads busy) */
    if (rows >= 64) ffma_block<4, 4, FULL_UNROLL>(sA, sB, cblk, rows, cblk_ok);
    else if (rows >= 32) ffma_block<2, 4, FULL_UNROLL>(sA, sB, cblk, rows, cblk_ok);
    else if (rows >= 16) ffma_block<2, 2, FULL_UNROLL>(sA, sB, cblk, rows, cblk_ok);
    else ffma_block<1, 2, FULL_UNROLL>(sA, sB, cblk, rows, cblk_ok);
  }
  __syncthreads();          /* every stage is free for the next body */
  return ok;
}

/* Dynamic shared memory a CTA asks for when P CTAs share an SM. */
__host__ __device__ constexpr uint32_t body_smem_bytes(int P) { return P == 2 ? SmemCfg<2>::dyn_bytes : LK_TC_SMEM; }

}  // namespace lk
#endif
