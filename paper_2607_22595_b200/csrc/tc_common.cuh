// Thin wrappers around the sm_100a instructions the tensor-core kernels of this library share:
// mbarriers with bounded waits, TMA tile loads (never multicast), shared-memory and instruction
// descriptors of tcgen05.mma (kind::f16 and kind::f8f6f4, operands K-major with the 128-byte swizzle), commit,
// fences, and the 32-lane x 32-column tensor-memory load.
#pragma once

#include <cuda.h>
#include <stdint.h>

#include "mix.h"

namespace mix {
namespace tc {

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
// `on` in this and the other instructions below that one thread issues: only where it is not 0 (see elect_one).
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes, unsigned on = 1u) {
  asm volatile("{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %2, 0;\n\t@e mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}"
               ::"r"(bar), "r"(bytes), "r"(on) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// The same without waiting at all: has the phase completed?
__device__ __forceinline__ unsigned mbar_test(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}

// Bounded wait.  Returns false if the wait ran longer than *cap_p clock cycles (the caller's CTA
// then raises MIX_STATUS_WAIT_TIMEOUT through `status` and sets *abort_flag) or if another role of
// the CTA already gave up.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned parity, volatile int* abort_flag,
                                                  const long long* cap_p, unsigned* status) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long cap = *cap_p;                 // read only on the slow path
  const long long t0 = clock64();
  unsigned spins = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++spins & 255u) == 0u) {
      if (*abort_flag) return false;
      if (clock64() - t0 > cap) {
        *abort_flag = 1;
        atomicOr(status, MIX_STATUS_WAIT_TIMEOUT);
        return false;
      }
    }
  }
  return true;
}

// The same by a whole warp, which gets one answer.
__device__ __forceinline__ bool mbar_wait_bounded_warp(unsigned bar, unsigned parity, volatile int* abort_flag,
                                                       const long long* cap_p, unsigned* status) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const long long cap = *cap_p;
  const long long t0 = clock64();
  unsigned spins = 0;
  while (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) {
    if ((++spins & 255u) == 0u) {
      if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
      if (__any_sync(0xffffffffu, clock64() - t0 > cap)) {
        *abort_flag = 1;
        if ((threadIdx.x & 31) == 0) atomicOr(status, MIX_STATUS_WAIT_TIMEOUT);
        return false;
      }
    }
  }
  return true;
}

// One lane of a converged warp, the same one every time.  A loop that issues copies or tensor-core instructions is run by the
// whole warp with this around the instructions themselves: their operands then live in uniform registers.  Inside a branch that
// one lane has taken each operand is moved there first, instruction by instruction -- 328 cycles to issue the four tcgen05.mma
// and the commit of a k-block.
__device__ __forceinline__ unsigned elect_one() {
  unsigned one;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
  return one;
}
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }

__device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar, unsigned on = 1u) {
  asm volatile(
      "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %5, 0;\n\t"
      "@e cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n\t}"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar), "r"(on)
      : "memory");
}

// The same for data that is read once (or by its readers at the same time) and larger than L2 -- a stream of weights: its
// lines are the first to be evicted, so that what the kernels around it share (their code among it) stays in L2.
__device__ __forceinline__ unsigned long long l2_evict_first() {
  unsigned long long p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ void tma_load_2d_hint(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar, unsigned long long policy,
                                                 unsigned on = 1u) {
  asm volatile(
      "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %6, 0;\n\t"
      "@e cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;\n\t}"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar), "l"(policy), "r"(on)
      : "memory");
}

// K-major operand tile, 128-byte swizzle: rows of 64 bf16 (128 B), 8-row groups 1024 B apart.
__device__ __forceinline__ unsigned long long umma_desc(unsigned smem_addr) {
  unsigned long long d = 0;
  d |= (unsigned long long)((smem_addr & 0x3FFFFu) >> 4);   // start address, 16-byte units
  d |= (unsigned long long)1 << 16;                         // leading byte offset (unused when swizzled)
  d |= (unsigned long long)(1024 >> 4) << 32;               // stride byte offset between 8-row groups
  d |= (unsigned long long)1 << 46;                         // descriptor version (sm_100)
  d |= (unsigned long long)2 << 61;                         // 128-byte swizzle
  return d;
}

// kind::f16 instruction descriptor: D fp32, A and B bf16, both K-major, M x N.
__host__ __device__ constexpr unsigned idesc_f16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(m >> 4) << 24);
}

__device__ __forceinline__ void umma_f16(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned idesc,
                                         unsigned accumulate, unsigned on = 1u) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(on)
      : "memory");
}
// kind::f8f6f4 with both operands E4M3 (format code 0), D fp32, both K-major: one instruction takes
// K = 32 elements = 32 bytes, so a 128-byte swizzled row holds four steps (bf16: 16 elements, same bytes).
__host__ __device__ constexpr unsigned idesc_e4m3(int m, int n) {
  return (1u << 4) | ((unsigned)(n >> 3) << 17) | ((unsigned)(m >> 4) << 24);
}
__device__ __forceinline__ void umma_e4m3(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned idesc,
                                          unsigned accumulate, unsigned on = 1u) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(on)
      : "memory");
}
__device__ __forceinline__ void umma_commit(unsigned bar, unsigned on = 1u) {
  asm volatile("{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %1, 0;\n\t@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
               ::"r"(bar), "r"(on) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(unsigned taddr, float* v) {
  unsigned* r = reinterpret_cast<unsigned*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld8(unsigned taddr, float (&v)[8]) {
  unsigned r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Contiguous bytes into shared memory (both addresses on 16 bytes, a multiple of 16), counted on an mbarrier.
__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// ---- CTA pairs (a cluster of two CTAs working on one 256-row tile with tcgen05 cta_group::2) ----
// Rank of this CTA in its cluster; the shared::cluster address of the same variable in CTA `rank` of the cluster;
// a cluster-wide barrier; an arrival on an mbarrier that may live in the peer CTA.
__device__ __forceinline__ unsigned cluster_ctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned mapa_cluster(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(unsigned cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// Tile load of one CTA of a pair: the data lands in THIS CTA's shared memory, the completion bytes are counted on
// a barrier given by its shared::cluster address, which may be the peer's (the pair's leader waits on one barrier
// for both halves of a stage).  No multicast: each CTA fetches its own half.
__device__ __forceinline__ void tma_load_2d_pair(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar_cluster, unsigned on = 1u) {
  asm volatile(
      "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %5, 0;\n\t"
      "@e cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n\t}"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar_cluster), "r"(on)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair_hint(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar_cluster,
                                                      unsigned long long policy, unsigned on = 1u) {
  asm volatile(
      "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %6, 0;\n\t"
      "@e cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;\n\t}"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar_cluster), "l"(policy), "r"(on)
      : "memory");
}
// One instruction of the pair: M = 256 (rows 0..127 from the A tile in the leader's shared memory, 128..255 from
// the peer's, accumulators in each CTA's own tensor memory), N = 256 with each CTA's shared memory holding 128 of
// the B rows.  Issued by one thread of the leader CTA.
__device__ __forceinline__ void umma_f16_pair(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned idesc,
                                              unsigned accumulate, unsigned on = 1u) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(on)
      : "memory");
}
__device__ __forceinline__ void umma_e4m3_pair(unsigned d_tmem, unsigned long long a, unsigned long long b, unsigned idesc,
                                               unsigned accumulate, unsigned on = 1u) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(on)
      : "memory");
}
// Arrives, once the instructions issued so far have completed, on the barrier at this offset in BOTH CTAs of the pair.
__device__ __forceinline__ void umma_commit_pair(unsigned bar, unsigned on = 1u) {
  const unsigned short mask = 3;
  asm volatile("{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %2, 0;\n\t"
               "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}"
               ::"r"(bar), "h"(mask), "r"(on)
               : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(unsigned smem_slot, unsigned cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_slot), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(unsigned base, unsigned cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}

__device__ __forceinline__ void tmem_alloc(unsigned smem_slot, unsigned cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_slot), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(unsigned base, unsigned cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}

}  // namespace tc
}  // namespace mix
