// CTA-pair forms of the tensor-core primitives (tcgen05 cta_group::2), shared by the kernels on pairs: CTAs 2 i and 2 i + 1
// of a cluster work on one accumulator tile, the even one (the leader) issues the MMAs, the copies of both signal its barrier.
#pragma once

#include "common.cuh"
#include "tmap.h"

namespace phyai {

constexpr uint32_t LEADER_MASK = 0xFEFFFFFFu;     // clears the lowest CTA-rank bit of a shared::cluster address

// rows of 64 bf16 from `row` on (the map's box high), into this CTA's shared memory
__device__ __forceinline__ void tma2d(uint32_t dst, const CUtensorMap* map, int row, uint32_t bar_leader) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(bar_leader)
      : "memory");
}
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
__device__ __forceinline__ void umma2_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrives on the barrier at this offset in the CTAs of `mask` once every MMA issued so far has completed
__device__ __forceinline__ void umma2_commit(uint32_t bar, uint32_t mask = 3) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"((uint16_t)mask)
               : "memory");
}
__device__ __forceinline__ void tmem_alloc2(uint32_t slot_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// this CTA's shared address, at CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// arrives on a barrier of this or another CTA of the cluster.  (Release at CTA scope: for arrivals that announce tensor memory, which is
// fenced by tcgen05.fence, or copies that the barrier counts itself.  At cluster scope the arrival of a softmax warp took 1500
// clocks per key tile, between the probabilities and their product.)
__device__ __forceinline__ void remote_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// The same for stores to shared memory (each behind the writer's own proxy fence) that the leader's MMAs read in this CTA: the release
// reaches the leader, whose MMA warp acquires it with pair_acquire on the completed phase.
__device__ __forceinline__ void remote_arrive_stores(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void pair_acquire(uint32_t bar, uint32_t parity) {
  uint32_t done;      // (the phase is complete, or the call has been given up)
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
}
// A operand in tensor memory
__device__ __forceinline__ void umma2_ts(uint32_t d, uint32_t ta, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d), "r"(ta), "l"(db), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void pair_sync() {      // every thread of every CTA of the cluster
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

}  // namespace phyai
