// Two-CTA building blocks (sm_100a, cta_group::2): a cluster of two CTAs on neighbouring SMs issues products of M = 256, each
// CTA holding 128 accumulator rows, its own half of A and half of B.  Against two single-CTA products of M = 128 an SM reads
// 8 KB of operands instead of 12 KB per 128 cycles, and B is fetched and stored once for both.
//   * The CTA of even rank (the leader) issues the products and owns the "operands have arrived" barriers; the loads of both
//     CTAs signal there.
//   * Commits signal the barrier at the same offset in both CTAs.
//   * Nothing is read through multicast loads.
#pragma once

#include "sm100.cuh"

namespace cafeq {

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}
// address of this CTA's shared variable in the CTA of the given rank
__device__ __forceinline__ uint32_t cluster_addr(uint32_t saddr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
  return a;
}
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
// Arrival at a barrier of either CTA after stores to shared memory that the other CTA's products read: releases them at the scope of
// the cluster, and the barrier is awaited with mbar_wait_pair.  It also waits until the thread's global stores have landed.
__device__ __forceinline__ void mbar_arrive_pair(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// Arrival after reads of tensor memory only (ordered by the tcgen05 fences): CTA scope.  With the scope of the cluster it waits for
// the thread's global stores, 2100 cycles a tile in the transform pass.
__device__ __forceinline__ void mbar_arrive_pair_tmem(uint32_t addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
struct PairAcquire {
  static __device__ __forceinline__ uint32_t try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok;
  }
};
// bounded wait for arrivals of both CTAs (mbar_arrive_pair)
__device__ __forceinline__ bool mbar_wait_pair(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status) {
  return mbar_wait<PairAcquire>(bar, parity, abort_flag, status);
}

// Whether either CTA of the pair saw a raised status word: one answer for both (a CTA that left alone would leave the other
// waiting on its barriers).  Also the point from which both CTAs' barriers may be signalled.  vote: a word of shared memory.
// Called by all threads of both CTAs; after a `true` every thread has to return (the peer may not be read any more).
__device__ __forceinline__ bool pair_stopped(bool raised, uint32_t* vote) {
  const int mine = __syncthreads_or(raised);
  if (threadIdx.x == 0) *vote = (uint32_t)(mine != 0);
  cluster_sync();
  const bool stop = ld_cluster_u32(cluster_addr(smem_u32(vote), cluster_rank() ^ 1u)) != 0u || mine != 0;
  if (stop) cluster_sync();
  return stop;
}

__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free_pair(uint32_t base, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}
// the barrier at this offset in both CTAs, when the products issued so far are done
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"((uint16_t)3)
               : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "mov.b64 a, {%1, %5};\n\tmov.b64 b, {%2, %5};\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(a_lo), "r"(b_lo), "r"(idesc), "r"(accumulate), "n"(UMMA_DESC_HI)
      : "memory");
}
// a load into this CTA's shared memory that signals `bar`, a barrier of either CTA (cluster address)
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_pair_hint(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(bar), "l"(pol)
      : "memory");
}

// launch of a grid of CTA pairs
template <typename... P, typename... A>
static inline void launch_pairs_if(bool overlap, void (*kernel)(P...), int pairs, int threads, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace cafeq
