// tma.cuh -- TMA tensor-map loads, mbarriers with bounded waits, and programmatic
// dependent launch control, as inline PTX for sm_103a.
#pragma once
#include <cuda.h>
#include <cstdint>

namespace hscale {

// Upper bound on polls of one mbarrier phase.  try_wait blocks for a hardware-chosen
// interval per poll (3.8 us on a GB300), so this is about a minute; a wait that runs out reports an
// error instead of hanging the GPU.
//
// A build with HSCALE_STARVED_BLOCK = b (the failure tests') has a limit of a few milliseconds, and in
// it mbar_wait_acc, the epilogues' wait for an accumulator, runs out at once in block b.
#ifndef HSCALE_STARVED_BLOCK
#define HSCALE_STARVED_BLOCK -1
#endif
constexpr int kStarvedBlock = HSCALE_STARVED_BLOCK;
constexpr uint32_t kMbarPollLimit = kStarvedBlock < 0 ? 1u << 24 : 1u << 10;

// Device-wide error word of this library (bit flags, sticky until read by the host).
constexpr uint32_t kErrMbarTimeout = 1u;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// make initialised barriers visible to the async (TMA) proxy and the cluster
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

// Wait for the phase with the given parity to complete; false once `limit` polls ran out.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t limit) {
  const uint32_t a = smem_addr(bar);
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  return mbar_wait_bounded(bar, parity, kMbarPollLimit);
}

__device__ __forceinline__ bool mbar_wait_acc(uint64_t* bar, uint32_t parity) {
  return (kStarvedBlock < 0 || (int)blockIdx.x != kStarvedBlock) && mbar_wait(bar, parity);
}

// The loads that a ring's producer has issued land before the CTA's shared memory may go away; after a
// wait that ran out nobody else waits for them.  (s, parity): the producer's position, the stage it
// would fill next and the parity of its wait for that one.  The stages before s were last filled in
// this turn of the ring, those from s on in the turn before (or never: a fresh barrier passes).
__device__ __forceinline__ void ring_drain(uint64_t* full, int stages, uint32_t s, uint32_t parity) {
  for (int t = 0; t < stages; ++t) mbar_wait(&full[t], t < (int)s ? parity ^ 1u : parity);
  __syncwarp();
}

// One lane of the (converged) warp.  The loops that issue TMA loads and MMAs run in a whole warp
// and only the instruction itself in the elected lane: their operands must be in uniform
// registers, and values computed by a single thread have to be moved there one by one (about 85
// cycles an MMA, measured).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// A whole warp waits; the same answer in every lane.
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity));
}
// The value of lane 0, which the compiler then knows to be uniform.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __shfl_sync(0xFFFFFFFFu, v, 0); }

// 2-D tiled TMA load of one box into this CTA's shared memory, completing on `bar`.
// c0 is the innermost coordinate (elements); c0 * element size must be a multiple of 16.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int32_t c0, int32_t c1,
                                            uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_addr(bar)), "l"(policy)
      : "memory");
}

// The same with a 3-D box.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int32_t c0, int32_t c1, int32_t c2,
                                            uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_addr(bar)), "l"(policy)
      : "memory");
}

// The same without a policy.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int32_t c0, int32_t c1, int32_t c2,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_addr(bar))
      : "memory");
}

// Generic-proxy writes to shared memory become visible to the async proxy (TMA, tcgen05).
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// L2 policy for data read exactly once
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// Programmatic dependent launch: let the next kernel on the stream start its prologue,
// and (in that kernel) wait until this one has finished and its writes are visible.  A kernel
// that waits takes what the kernel before it writes through plain pointers: __restrict__ would let the
// compiler load it before the wait, or past the coherent caches.
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait_primary() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace hscale
