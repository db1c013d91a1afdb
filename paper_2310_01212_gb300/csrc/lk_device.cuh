/*
 * lk_device.cuh -- device primitives: memory-model loads/stores at system and
 * GPU scope, %smid / %globaltimer, bounded spin back-off, TMA bulk copies
 * with mbarrier completion.  All inline PTX written for sm_103a.
 */
#ifndef LK_DEVICE_CUH
#define LK_DEVICE_CUH
#include <stdint.h>

namespace lk {

/* ---- bounds checks of the checking build (-DLK_DEBUG_BOUNDS) ------------
 * LK_INB(cond, site) guards one access: in the checking build a false
 * `cond` counts a violation, records the first site and returns false, so
 * the caller skips the access instead of faulting; in the product build it
 * is `true` and `cond` is not evaluated.  Sites name the access path. */
enum : uint32_t {
  LK_OOB_SHARE = 1,        /* a CTA's or warp's share outside the operand       */
  LK_OOB_STREAM_LOAD = 2,  /* a staged chunk outside the share, or misaligned   */
  LK_OOB_STREAM_SMEM = 3,  /* a stage outside the streaming region              */
  LK_OOB_STORE = 4,        /* an element store outside the share                */
  LK_OOB_HIST_COUNTER = 5, /* a histogram counter outside the work region      */
  LK_OOB_GEMM_LOAD = 6,    /* a GEMM tile or row block outside the operands     */
  LK_OOB_GEMM_STORE = 7,   /* a GEMM store outside the output tile              */
  LK_OOB_GEMM_SMEM = 8,    /* a GEMM stage, operand buffer or TMEM column out   */
};
#ifdef LK_DEBUG_BOUNDS
__device__ unsigned long long g_lk_oob_count;
__device__ unsigned int g_lk_oob_site;
__device__ __forceinline__ bool lk_inb(bool ok, uint32_t site) {
  if (!ok && atomicAdd(&g_lk_oob_count, 1ull) == 0ull) atomicExch(&g_lk_oob_site, site);
  return ok;
}
__device__ __forceinline__ bool lk_oob_seen() { return *(volatile unsigned long long*)&g_lk_oob_count != 0ull; }
#define LK_INB(cond, site) ::lk::lk_inb((cond), (site))
#else
#define LK_INB(cond, site) true
#endif

__device__ __forceinline__ uint64_t gtime() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t smid() {
  uint32_t s;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(s));
  return s;
}

/* system scope: host-mapped words shared with the host CPU */
__device__ __forceinline__ uint64_t ld_acquire_sys(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.acquire.sys.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t ld_relaxed_sys(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.sys.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_sys(uint64_t* p, uint64_t v) {
  asm volatile("st.release.sys.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed_sys(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.sys.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed_sys32(int32_t* p, int32_t v) {
  asm volatile("st.relaxed.sys.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void red_release_sys_add(uint32_t* p, uint32_t v) {
  asm volatile("red.release.sys.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t cas_relaxed_sys(uint32_t* p, uint32_t cmp, uint32_t v) {
  uint32_t old;
  asm volatile("atom.relaxed.sys.cas.b32 %0, [%1], %2, %3;" : "=r"(old) : "l"(p), "r"(cmp), "r"(v) : "memory");
  return old;
}

/* GPU scope: cluster-internal relay words in device memory (L2) */
__device__ __forceinline__ uint64_t ld_acquire_gpu(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.acquire.gpu.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_acquire_gpu32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(uint64_t* p, uint64_t v) {
  asm volatile("st.release.gpu.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t atom_add_acq_rel_gpu(uint32_t* p, uint32_t v) {
  uint32_t old;
  asm volatile("atom.acq_rel.gpu.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ uint64_t ld_relaxed_gpu(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int32_t ld_relaxed_gpu_s32(const int32_t* p) {
  int32_t v;
  asm volatile("ld.relaxed.gpu.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_relaxed_gpu_add_s32(int32_t* p, int32_t v) {
  asm volatile("red.relaxed.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

/* Programmatic dependent launch: a kernel launched that way may start while
 * the one before it in the stream still runs; it waits here until that one has
 * finished and its writes are visible.  Both are no-ops otherwise. */
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

/* Named CTA barriers (id 1..15; 0 is __syncthreads): `threads` arrivals open
 * one; bar_sync waits for it, bar_arrive only counts in.  Whole warps only. */
__device__ __forceinline__ void bar_sync(uint32_t id, uint32_t threads) {
  asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t id, uint32_t threads) {
  asm volatile("barrier.cta.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

/* bar_sync that also returns the AND of every participant's v. */
__device__ __forceinline__ bool bar_sync_and(uint32_t id, uint32_t threads, bool v) {
  uint32_t out;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.u32 pi, %1, 0;\n\t"
      "barrier.cta.red.and.pred po, %2, %3, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(out)
      : "r"((uint32_t)v), "r"(id), "r"(threads)
      : "memory");
  return out != 0;
}

/* Exponential back-off between polls.  base == 0 spins without sleeping. */
struct Backoff {
  uint32_t ns, cap;
  __device__ __forceinline__ Backoff(uint64_t base, uint64_t cap_) : ns((uint32_t)base), cap((uint32_t)cap_) {}
  __device__ __forceinline__ void pause() {
    if (ns) {
      __nanosleep(ns);
      ns = ns * 2 > cap ? cap : ns * 2;
    }
  }
};

/* ---- TMA bulk copy (non-multicast) into this CTA's shared memory ------- */
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
/* global -> shared bulk copy; src and dst 16-byte aligned, bytes % 16 == 0 */
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
/* Bounded wait for an mbarrier phase; false if the deadline passed. */
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t deadline) {
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 15) == 15 && gtime() > deadline) return false;
  }
}

/* shared -> global bulk copy (the async proxy reads shared memory) */
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
/* every committed bulk store has finished reading shared memory */
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
/* every committed bulk store has completed */
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

/* ---- 5th-generation tensor cores (tcgen05) and tensor memory ---------- */
/* Allocate `ncols` (power of two, >= 32) TMEM columns; one whole warp
 * executes it and the base address lands in *dst (shared memory). */
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(dst)), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

/* Shared-memory matrix descriptor, 128-byte swizzle (bits 61-63 = 2): start
 * address, leading and stride byte offsets, bits 46-47 the descriptor version
 * (1).  Atoms are 8 rows of 128 bytes (1 KB, on 1 KB boundaries).  K-major:
 * a row holds 64 k of one m, sbo = byte distance between groups of 8 m (lbo
 * unused).  MN-major: a row holds 64 n of one k, lbo = byte distance between
 * blocks of 64 n, sbo = between groups of 8 k. */
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3fffu) | ((uint64_t)((lbo >> 4) & 0x3fffu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3fffu) << 32) | (1ull << 46) | (2ull << 61);
}

/* True on one lane of a converged warp.  Tensor-core instructions take their
 * operands from uniform registers: issued under this predicate in a
 * warp-uniform branch they cost about 32 clocks each; under a thread-index
 * test, where the compiler must assume any lane, 51 (one issuing thread, a
 * chain of M = 64, N = 64 MMAs). */
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(p)
      :
      : "memory");
  return p != 0;
}

/* D[tmem] (+)= A[smem] * B[smem]^T, kind::f16 (both operands bf16 here), issued by one thread. */
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

/* Arrive on mbarrier `bar` once every MMA this thread issued has completed. */
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}

/* 16 TMEM lanes from ta's (and tb's), 32 consecutive fp32 columns each: of
 * columns 8 j .. 8 j + 7, thread t holds columns 2 (t % 4), + 1 of lane t / 4
 * in v[4 j], v[4 j + 1] and of lane t / 4 + 8 in v[4 j + 2], v[4 j + 3]. */
__device__ __forceinline__ void tmem_ld_16x256b_x4_2(uint32_t ta, uint32_t tb, float* v, float* w) {
  uint32_t r[16], q[16];
#define LK_TMEM_LD(x, taddr)                                                                                          \
  asm volatile(                                                                                                       \
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "     \
      "%15}, [%16];"                                                                                                  \
      : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7]), "=r"(x[8]),   \
        "=r"(x[9]), "=r"(x[10]), "=r"(x[11]), "=r"(x[12]), "=r"(x[13]), "=r"(x[14]), "=r"(x[15])                      \
      : "r"(taddr)                                                                                                    \
      : "memory")
  LK_TMEM_LD(r, ta);
  LK_TMEM_LD(q, tb);
#undef LK_TMEM_LD
  /* the registers are valid only after the wait: tying them to it keeps
   * every use of them below it */
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]), "+r"(q[6]),
                 "+r"(q[7]), "+r"(q[8]), "+r"(q[9]), "+r"(q[10]), "+r"(q[11]), "+r"(q[12]), "+r"(q[13]),
                 "+r"(q[14]), "+r"(q[15])
               :
               : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    v[i] = __uint_as_float(r[i]);
    w[i] = __uint_as_float(q[i]);
  }
}

/* streaming 128-bit loads / stores (coherent path; no .nc: a persistent
 * kernel outlives the writes other kernels make to its inputs) */
__device__ __forceinline__ int4 ld_stream(const int4* p) { return __ldcs(p); }
__device__ __forceinline__ float4 ld_stream(const float4* p) { return __ldcs(p); }
__device__ __forceinline__ uint4 ld_stream(const uint4* p) { return __ldcs(p); }
__device__ __forceinline__ void st_stream(int4* p, int4 v) { __stcs(p, v); }
__device__ __forceinline__ void st_stream(float2* p, float2 v) { __stcs(p, v); }

}  // namespace lk
#endif
