// Bulk asynchronous global->shared copies (TMA, untiled form) completed on an mbarrier, with bounded waits.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace tj {

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t arrivals) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(arrivals) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

// dst and src 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

// the same copy with an L2 eviction policy for the lines it reads (e.g. l2_evict_last_policy() for data every block re-reads)
__device__ __forceinline__ unsigned long long l2_evict_last_policy() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void bulk_copy_g2s_keep(void* dst, const void* src, uint32_t bytes, uint64_t* bar, unsigned long long policy) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Polls before a wait gives up.  A build with 0 makes every bounded wait run out at once: how the tests reach what follows then.
#ifndef TJ_WAIT_POLLS
#define TJ_WAIT_POLLS (1 << 22)
#endif

// Waits for the phase with the given parity; gives up after a fixed number of polls and reports false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
#pragma unroll 1
  for (int i = 0; i < TJ_WAIT_POLLS; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// The wait of a block that gives up for what it still has in flight (bulk copies, matrix instructions): none of it may arrive after
// the block has handed its shared memory to another.  Bounded as well, but whatever TJ_WAIT_POLLS says.
__device__ __forceinline__ void mbar_settle(uint64_t* bar, uint32_t parity) {
#pragma unroll 1
  for (int i = 0; i < (1 << 22); ++i)
    if (mbar_try_wait(bar, parity)) return;
}

// per-thread asynchronous copies of 16 (both addresses aligned) or 4 bytes, waited for by groups
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
// this thread's arrival at `bar` (one of the expected) when its copies so far have landed
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Start of a kernel launched by launch_chained: waits until the kernel before it has finished and its writes are visible.
// A kernel that allocates tensor memory calls this after the allocation: a successor resident on the same SM may ask for
// tensor memory too, and must find this block's share already taken.
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the stream become resident once every block has come this far (or left).  Short kernels call it
// right after chain_begin(); kernels that fill the SMs leave it to their blocks' exits: a successor placed while they run
// would crowd onto the few SMs that are idle (the FP32 learner lost 10 % to that).
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// all threads of the cluster's blocks meet (arrive has release, wait acquire semantics over distributed shared memory)
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Arrival at the barrier at this block's address `bar` in block `rank` of the cluster, and the wait for arrivals from another block.  They
// hand over what the arriving block has in its own shared memory (and, with the tcgen05 fences, its reads of tensor memory): a release and
// an acquire at cluster scope, of shared memory alone.  The same without that restriction also waits for the record stores in flight
// (65,536 CartPole envs, hidden 256, 128 steps: 3.25 ms; 2.58 like this).
__device__ __forceinline__ void mbar_arrive_cluster(uint64_t* bar, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(bar)), "r"(rank));
  asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(a) : "memory");
}
__device__ __forceinline__ void cluster_acquire() { asm volatile("fence.acquire.sync_restrict::shared::cluster.cluster;" ::: "memory"); }
__device__ __forceinline__ bool mbar_try_wait_relaxed(uint64_t* bar, uint32_t parity) {    // cluster_acquire() has to follow
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// a float at this block's shared-memory address `p` in block `rank` of the cluster
__device__ __forceinline__ float cluster_load_f32(const float* p, uint32_t rank) {
  uint32_t a;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ void cluster_store_f32(float* p, uint32_t rank, float v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

// One thread queues `bytes` (multiple of 16) in chunks; the barrier must expect the same total.
__device__ __forceinline__ void bulk_copy_chunks(void* dst, const void* src, size_t bytes, uint64_t* bar) {
  constexpr size_t kChunk = 16384;
  for (size_t o = 0; o < bytes; o += kChunk) {
    const size_t n = bytes - o < kChunk ? bytes - o : kChunk;
    bulk_copy_g2s(static_cast<char*>(dst) + o, static_cast<const char*>(src) + o, (uint32_t)n, bar);
  }
}

}  // namespace tj
