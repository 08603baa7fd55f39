// Blackwell (sm_103a) tensor-core building blocks written as inline PTX:
// mbarriers with bounded waits, TMA tile loads, tcgen05 shared-memory and
// instruction descriptors, tcgen05.mma / commit, TMEM allocation and loads.
#pragma once

#include <cuda.h>
#include <stdint.h>

#include "exa_internal.cuh"

namespace exa {
namespace tc {

// Longest a single wait may take before the kernel gives up (SM clock cycles, ~1 s).
constexpr long long kWaitCycles = 2000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for the phase with the given parity to complete.  Gives up after
// kWaitCycles or as soon as *abort is set by another role; returns false then.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort) {
  if (mbar_try_wait(b, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try_wait(b, parity)) return true;
    if (*abort) return false;
    if (clock64() - t0 > kWaitCycles) return false;
  }
}

// A flag in shared memory between warps of one CTA: what was written before post is seen after await, which polls (a
// few tens of cycles; an mbarrier wait takes longer to wake).  `polls` bounds a thread's waits together: once it has run
// out (~0.3 s from kFlagPolls) they all return at once, and report_waits puts that into the status.
constexpr int kFlagPolls = 1 << 24;
__device__ __forceinline__ void post(int* flag, int v) {
  asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"(smem_u32(flag)), "r"(v) : "memory");
}
__device__ __forceinline__ void await(const int* flag, int v, int& polls) {
  int got;
  do {
    asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(got) : "r"(smem_u32(flag)) : "memory");
  } while (got != v && --polls > 0);
}
__device__ __forceinline__ void report_waits(int polls, DevStatus* st, int site) {
  if (polls <= 0 && atomicExch(&st->timeout, 1) == 0) st->timeout_where = site;
}

// L2 policy for operand tiles that later tiles of the same launch read again: kept in L2
// ahead of the streamed FP64 C tiles (which are loaded and stored with evict-first hints).
__device__ __forceinline__ uint64_t l2_evict_last_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__device__ __forceinline__ void tma_load_2d_hint(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y,
                                                 uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, "
      "%4}], [%2], %5;" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(smem_u32(bar)), "r"(x), "r"(y), "l"(pol)
      : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)map) : "memory");
}

// tcgen05 shared-memory matrix descriptor for a K-major operand laid out by a
// TMA load with 128-byte swizzling: rows of 128 bytes, 8-row (1024-byte)
// swizzle atoms stacked along M/N (stride 1024 bytes).  Fields: start address
// >> 4 in bits [0,14), leading offset (unused here) [16,30), stride offset >> 4
// [32,46), the fixed value 1 in [46,48), swizzle mode in [61,64) (2 = 128B).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Shared-memory descriptor of a K-major operand without swizzling: 8-row core matrices of 128 bytes, the two of
// a 16-column step 128 bytes apart (leading offset), 8-row groups 256 bytes apart (stride offset).
__device__ __forceinline__ uint64_t sdesc_flat(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(256 >> 4) << 32) |
         ((uint64_t)1 << 46);
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// An FP32 integer, |a| <= 2^24, by additions: the multiples of 4 from a + 1.5 2^25, then the rest.
__device__ __forceinline__ int f32_to_int(float a) {
  const float u = a + 50331648.0f;
  const float rest = a - (u - 50331648.0f);
  return 4 * (__float_as_int(u) - 0x4C400000) + (__float_as_int(rest + 12582912.0f) - 0x4B400000);
}

// Instruction descriptor for kind::tf32 / kind::f16: D format F32 (bits 4-5 = 1),
// A/B formats in bits [7,10) / [10,13) (BF16 = 1, TF32 = 2), both K-major,
// N >> 3 in bits [17,23), M >> 4 in bits [24,29).
constexpr uint32_t kFmtBF16 = 1;
constexpr uint32_t kFmtTF32 = 2;
__host__ __device__ constexpr uint32_t idesc(uint32_t fmt, int M, int N) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}

// Arrive once on `bar` when every tcgen05 operation issued so far by this thread completes.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Whole-warp TMEM allocation; the base address is written to *dst (shared).
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// 4 consecutive 32-bit columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// 16 consecutive 32-bit columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------------------
// CTA pairs (cluster of two CTAs on two SMs, tcgen05 .cta_group::2).  The MMA
// of the even CTA (the leader) reads A and B halves from both CTAs' shared
// memory and writes each CTA's accumulator rows into that CTA's TMEM.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Shared::cluster address of the object at local shared address `a` in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

// Arrive on an mbarrier given by its shared::cluster address (possibly in the peer CTA).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// 2-D TMA tile load into this CTA's shared memory whose byte count completes on the
// mbarrier at shared::cluster address `bar` (in either CTA of the pair), with an L2 policy.
__device__ __forceinline__ void tma_load_2d_pair_hint(void* dst, const CUtensorMap* map, uint32_t bar, int x, int y,
                                                      uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes.cta_group::2.L2::cache_hint [%0], "
      "[%1, {%3, %4}], [%2], %5;" ::"r"(smem_u32(dst)),
      "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y), "l"(pol)
      : "memory");
}

__device__ __forceinline__ void mma_tf32_pair(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}

// Arrive once on the mbarrier at local offset `bar` in every CTA of ctaMask when all
// tcgen05 operations issued so far by this thread complete.
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"(mask)
      : "memory");
}

// Pair-wide TMEM allocation: one warp of each CTA of the pair (same warp index) issues it.
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// ---------------------------------------------------------------------------
// Epilogue arithmetic on the integer pipe.  FP64 instructions issue at ~1.6 per
// clock per SM on this part, so per-element FP64 work in an epilogue costs more
// than the tile's tensor-core time; the conversions below use integer
// instructions only.
// ---------------------------------------------------------------------------

// FP32 bit pattern -> double, exact for normal values; zero and FP32 subnormals
// give a signed zero, infinities and NaNs stay infinities and NaNs.
__device__ __forceinline__ double f32_bits_to_f64(uint32_t u) {
  const uint32_t e = (u >> 23) & 0xFFu;
  const uint32_t sign = u & 0x80000000u;
  const uint32_t m = u & 0x7FFFFFu;
  const uint32_t de = (e == 0xFFu) ? 0x7FFu : e + 896u;  // rebias 127 -> 1023
  uint32_t hi = sign | (de << 20) | (m >> 3);
  uint32_t lo = m << 29;
  if (e == 0) {
    hi = sign;
    lo = 0;
  }
  return __hiloint2double((int)hi, (int)lo);
}

// V * 2^sh for an integer |V| < 2^53 (exactly representable): the double is built
// from V's bits; results below the normal range flush to zero.
__device__ __forceinline__ double i53_to_f64_scaled(long long V, int sh) {
  if (V == 0) return 0.0;
  const unsigned long long sgn = (unsigned long long)V & 0x8000000000000000ull;
  const unsigned long long M = V < 0 ? (unsigned long long)(-V) : (unsigned long long)V;
  const int lz = __clzll((long long)M);
  const unsigned long long frac = (M << (lz + 1)) >> 12;  // the bits below the leading one
  const long long be = (long long)(63 - lz) + 1023 + sh;
  if (be <= 0) return __longlong_as_double((long long)sgn);
  return __longlong_as_double((long long)(sgn | ((unsigned long long)be << 52) | frac));
}

}  // namespace tc
}  // namespace exa
