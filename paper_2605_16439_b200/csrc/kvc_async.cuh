// mbarrier + bulk-copy (TMA engine, 1-D) helpers for sm_100a.  Every wait is bounded: after
// WAIT_SPIN_LIMIT failed polls the caller records KVC_ERR_TIMEOUT in the device status word and
// leaves its loop, so a lost completion cannot hang the GPU.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace kvc {

// A try_wait on a barrier that does not complete comes back after about 7800 cycles (measured on B200), so 2^18 polls
// are about one second; a legitimate wait is far below a millisecond.
constexpr uint32_t WAIT_SPIN_LIMIT = 1u << 18;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count));
}
// makes mbarrier initialisation visible to the async (bulk copy) proxy
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}
// generic accesses to every state space before async-proxy accesses after it (a hand-over through global memory, both sides)
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;\n" ::: "memory"); }
// barrier among a subset of the CTA's warps (id 1..15; id 0 is __syncthreads)
__device__ __forceinline__ void named_barrier_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(nthreads) : "memory");
}
// producer / consumer use of a named barrier: `nthreads` counts arrivers and waiters together; arrivers do not block
__device__ __forceinline__ void named_barrier_arrive(int id, int nthreads) {
  asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(nthreads) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// one immediate look at the phase (no time-limited suspension as try_wait has)
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// true on completion, false if the spin limit ran out.  ROLLED: the loop is left rolled, which keeps the code around the wait small (three-kernel
// path, 16 x 8 blocks of n = 1024: 47.2 us a call unrolled, 46.0 rolled; cluster path, 26 calls it takes by default: 68.9 and 67.3 in the geometric
// mean).  The uniform one-kernel path takes 1 % less with the compiler's choice, the cluster path's text warps about 1 % (35 calls of 1000 to 3800 text
// rows 126.8 and 125.5, where with all waits unrolled they take 128.9; 30 x 10 blocks of n = 81, 3800 rows 71.1 and 67.8)
template <bool ROLLED = true>
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  if constexpr (ROLLED) {
#pragma unroll 1
    for (uint32_t i = 0; i < WAIT_SPIN_LIMIT; ++i)
      if (mbar_try_wait(bar, parity)) return true;
  } else {
    for (uint32_t i = 0; i < WAIT_SPIN_LIMIT; ++i)
      if (mbar_try_wait(bar, parity)) return true;
  }
  return false;
}

// global -> shared bulk copy; dst, src 16-byte aligned, bytes a multiple of 16; completion is
// signalled on `bar` as transaction bytes
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}

// ---- thread-block clusters: rank, a peer's shared-memory window, remote stores and mbarrier arrivals ----
__device__ __forceinline__ uint32_t cluster_ctarank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r)); return r; }
// address of the same shared-memory location in CTA `rank` of the cluster (a shared::cluster address)
__device__ __forceinline__ uint32_t map_to_cta(uint32_t local_saddr, uint32_t rank) {
  uint32_t r; asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(local_saddr), "r"(rank)); return r;
}
__device__ __forceinline__ void st_cluster_u32(uint32_t caddr, uint32_t v) { asm volatile("st.shared::cluster.u32 [%0], %1;\n" ::"r"(caddr), "r"(v) : "memory"); }
__device__ __forceinline__ void st_cluster_v4(uint32_t caddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(caddr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void st_cluster_f32(uint32_t caddr, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(caddr), "f"(v) : "memory"); }
__device__ __forceinline__ void st_cluster_f32x2(uint32_t caddr, float x, float y) { asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};\n" ::"r"(caddr), "f"(x), "f"(y) : "memory"); }
// one arrival on a peer's mbarrier; orders the calling CTA's earlier remote stores (after a CTA barrier) before it
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cbar) {
  asm volatile("fence.acq_rel.cluster;\n" ::: "memory");
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(cbar) : "memory");
}
// the arrival alone (release at cluster scope), for a caller that has fenced its warp's accesses itself
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cbar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(cbar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\n"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster_bounded(uint64_t* bar, uint32_t parity) {
#pragma unroll 1
  for (uint32_t i = 0; i < WAIT_SPIN_LIMIT; ++i)
    if (mbar_try_wait_cluster(bar, parity)) return true;
  return false;
}
// asynchronous stores into a peer's shared memory; their bytes are reported to the peer's barrier when they have landed
__device__ __forceinline__ void st_async_f32x2(uint32_t caddr, float x, float y, uint32_t cbar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];\n" ::"r"(caddr), "f"(x), "f"(y), "r"(cbar) : "memory");
}
__device__ __forceinline__ void st_async_f32x4(uint32_t caddr, const float4& v, uint32_t cbar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];\n"
               ::"r"(caddr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(cbar) : "memory");
}
// this CTA's shared memory -> a peer's, 16-byte aligned; completion on the peer's barrier
__device__ __forceinline__ void bulk_s2peer(uint32_t dst_caddr, uint32_t src_saddr, uint32_t bytes, uint32_t cbar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
               ::"r"(dst_caddr), "r"(src_saddr), "r"(bytes), "r"(cbar) : "memory");
}
// the two halves of cluster_sync_all
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
// every thread of every CTA of the cluster
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// every thread of every CTA of the cluster, diverged or not: no CTA leaves while a peer may still store into its
// shared memory or arrive on its barriers
__device__ __forceinline__ void cluster_exit_sync() {
  asm volatile("barrier.cluster.arrive.release;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory");
}

// programmatic dependent launch: wait for the preceding kernel of the stream to complete and flush;
// allow the next kernel of the stream to begin launching
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

}  // namespace kvc
