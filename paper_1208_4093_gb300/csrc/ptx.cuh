// Inline-PTX helpers for sm_103a: mbarriers and 1-D bulk (TMA) copies.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace hms {

// Programmatic dependent launch: dep_wait holds a CTA until the kernels before in
// the stream are complete and their writes visible (every thread of every CTA
// calls it before its first access to anything they write, and before any
// return, so that completion carries on from kernel to kernel); dep_launch lets
// the next kernel's CTAs be placed once all CTAs of this one have called it.
// Without effect in a kernel launched the ordinary way.
__device__ inline void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ inline void dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Cluster barrier in two halves, for the start of a kernel: a CTA may touch another
// one's shared memory only once that one runs, which is known when cluster_wait
// returns.  Every thread of the cluster calls both, cluster_arrive as early as it
// likes.  Orders no memory accesses.
__device__ inline void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ inline void cluster_wait() { asm volatile("barrier.cluster.wait;" ::: "memory"); }

__device__ inline uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ inline void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ inline void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Orders this thread's earlier shared-memory accesses before later async-proxy
// (bulk copy) accesses of the same memory.
// Global memory written by generic-proxy stores, then read by a bulk copy
// (async proxy): the writes must be ordered before the copy by this fence.
__device__ inline void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ inline void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ inline void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

// 1-D bulk copy global -> shared, completion counted on `bar` (bytes).
// dst, src 16-byte aligned; bytes a multiple of 16.
__device__ inline void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// 16 bytes global -> shared by the issuing thread, past L1; groups of them are
// waited for in order by the same thread.
__device__ inline void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ inline void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ inline bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for phase `parity` of `bar`: at most `limit` tries; false if
// it gave up.
constexpr uint32_t MBAR_WAIT_TRIES = 1u << 22;
__device__ inline bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t limit = MBAR_WAIT_TRIES) {
  for (uint32_t it = 0; it < limit; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

}  // namespace hms
