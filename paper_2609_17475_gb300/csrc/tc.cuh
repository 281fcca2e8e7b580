// tcgen05 (5th-generation tensor core) helpers: TMEM allocation, shared-memory
// matrix descriptors, instruction descriptors, MMA issue/commit and TMEM
// loads/stores (inline PTX for sm_103a).
#pragma once

#include "common.cuh"

namespace jfkv {
namespace tc {


// Shared-memory matrix descriptor, 128-byte swizzle (layout type 2), version 1.
// addr/lbo/sbo in bytes (16-byte granularity).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= 1ull << 46;
  d |= 2ull << 61;
  return d;
}

// Instruction descriptor, kind::f16 with f16 A/B and f32 accumulation.
// a_mn / b_mn: 0 = K-major, 1 = MN-major.
__host__ __device__ constexpr uint32_t idesc_f16_f32(int M, int N, int a_mn, int b_mn) {
  return (1u << 4) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Registers per thread of the executing warpgroup (every warp of it calls this).
template <int N>
__device__ __forceinline__ void setmaxnreg_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void setmaxnreg_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(N));
}

__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}

// ---- CTA pair (cluster of 2, cta_group::2) -------------------------------
// One warp of each CTA of the pair allocates; both receive the same address.
__device__ __forceinline__ void alloc2(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n"
               ::"r"(smem_u32(smem_dst)), "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n");
}

__device__ __forceinline__ void dealloc2(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols));
}

// 1 in one elected lane of the (converged) warp, 0 in the others.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(r));
  return r;
}

// Pair MMA, issued by one thread of CTA 0 (the one with leader != 0; the whole
// warp runs the issuing code, so its operands stay in uniform registers): M = 256, each CTA supplies (and
// receives in its TMEM) 128 rows of A and D and half of B's N columns, read
// from the same shared-memory offset in each CTA.
__device__ __forceinline__ void mma2_ts(uint32_t leader, uint32_t d_tmem, uint32_t a_tmem,
                                        uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
      : "memory");
}

// Pair MMA with both operands in shared memory (same offsets in each CTA):
// each CTA supplies 128 rows of A and half of B's N columns.
__device__ __forceinline__ void mma2_ss(uint32_t leader, uint32_t d_tmem, uint64_t a_desc,
                                        uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(leader)
      : "memory");
}

// The barrier at this shared offset in both CTAs arrives once the pair's
// tcgen05 ops issued so far by this thread are done.
__device__ __forceinline__ void commit2_both(uint32_t leader, uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;\n\t}\n" ::"r"(smem_u32(bar)), "h"((uint16_t)3), "r"(leader) : "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n"
               "barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Arrive on the mbarrier at this shared offset in CTA `rank` of the cluster
// (the own CTA included).  The data it publishes is this CTA's own shared
// memory (made visible to the tensor core by fence.proxy.async first) or its
// own TMEM (tcgen05.wait::st and tcgen05.fence::before_thread_sync first), so
// a CTA-scope release is enough: it orders the shared-memory stores before
// the arrive without draining the SM's outstanding global accesses, which a
// cluster-scope release waits for (measured: ~1,000 cycles per arrive in the
// prefill kernel under load).
__device__ __forceinline__ void arrive_cluster(uint64_t* bar, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(remote) : "r"(smem_u32(bar)), "r"(rank));
  asm volatile("mbarrier.arrive.release.cta.shared::cluster.b64 _, [%0];\n"
               ::"r"(remote) : "memory");
}

// The same with the address already mapped to CTA 0 (map_rank0), for loops
// whose barriers are an offset from one base.
__device__ __forceinline__ uint32_t map_rank0(uint32_t addr) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;\n" : "=r"(remote) : "r"(addr));
  return remote;
}
__device__ __forceinline__ void arrive_mapped(uint32_t remote) {
  asm volatile("mbarrier.arrive.release.cta.shared::cluster.b64 _, [%0];\n"
               ::"r"(remote) : "memory");
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;\n" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Bounded wait with cluster-scope acquire (for barriers other CTAs arrive on).
// Four polls to a step of the loop: the polls of waiting warps compete for
// issue slots with the warps they wait for.
#define JF_POLL(scope, hint)                                                                        \
  asm volatile(                                                                               \
      "{\n\t.reg .pred p;\n\t.reg .u32 c;\n\tmov.u32 c, %3;\n"                                 \
      "POLL:\n\t"                                                                             \
      "mbarrier.try_wait.parity.acquire." scope ".shared::cta.b64 p, [%1], %2" hint ";\n\t" \
      "@p bra DONE;\n\t"                                                                      \
      "mbarrier.try_wait.parity.acquire." scope ".shared::cta.b64 p, [%1], %2" hint ";\n\t" \
      "@p bra DONE;\n\t"                                                                      \
      "mbarrier.try_wait.parity.acquire." scope ".shared::cta.b64 p, [%1], %2" hint ";\n\t" \
      "@p bra DONE;\n\t"                                                                      \
      "mbarrier.try_wait.parity.acquire." scope ".shared::cta.b64 p, [%1], %2" hint ";\n\t" \
      "@p bra DONE;\n\t"                                                                      \
      "add.s32 c, c, -1;\n\tsetp.ne.s32 p, c, 0;\n\t@p bra POLL;\n"                           \
      "DONE:\n\tmov.u32 %0, c;\n\t}\n"                                                       \
      : "=r"(left) : "r"(addr), "r"(parity), "r"(steps) : "memory")

__device__ __forceinline__ bool wait_cluster_at(uint32_t addr, uint32_t parity,
                                                uint32_t steps = (1u << 20)) {
  uint32_t left;
  JF_POLL("cluster", "");
  return left != 0;
}
__device__ __forceinline__ bool wait_cta_at(uint32_t addr, uint32_t parity,
                                            uint32_t steps = (1u << 20)) {
  uint32_t left;
  JF_POLL("cta", "");
  return left != 0;
}
// For a producer that runs ahead: each poll may sleep for up to a microsecond.
__device__ __forceinline__ bool wait_cta_idle_at(uint32_t addr, uint32_t parity,
                                                 uint32_t steps = (1u << 18)) {
  uint32_t left;
  JF_POLL("cta", ", 1000");
  return left != 0;
}
#undef JF_POLL
__device__ __forceinline__ bool wait_cluster(uint64_t* bar, uint32_t parity,
                                             uint32_t steps = (1u << 20)) {
  return wait_cluster_at(smem_u32(bar), parity, steps);
}

#define JF_R8(i) "=r"(v[i]), "=r"(v[i + 1]), "=r"(v[i + 2]), "=r"(v[i + 3]), "=r"(v[i + 4]), \
                 "=r"(v[i + 5]), "=r"(v[i + 6]), "=r"(v[i + 7])

// 32 lanes x 32 columns of 32-bit words: thread i gets row (lane base + i).
__device__ __forceinline__ void ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : JF_R8(0), JF_R8(8), JF_R8(16), JF_R8(24)
      : "r"(taddr));
}

#define JF_W8(i) "r"(v[i]), "r"(v[i + 1]), "r"(v[i + 2]), "r"(v[i + 3]), "r"(v[i + 4]), \
                 "r"(v[i + 5]), "r"(v[i + 6]), "r"(v[i + 7])

__device__ __forceinline__ void st32(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
      "%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n"
      ::"r"(taddr), JF_W8(0), JF_W8(8), JF_W8(16), JF_W8(24)
      : "memory");
}

#undef JF_R8
#undef JF_W8

__device__ __forceinline__ void wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
}

}  // namespace tc
}  // namespace jfkv
