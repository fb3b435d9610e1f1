// Shared-memory staging primitives for sm_100a: mbarrier-tracked 1-D bulk
// copies (the TMA engine's untiled form; every copy is CTA-local, one source,
// one destination) and programmatic dependent launch.
//
// Every wait is bounded: after kSpinLimit unsuccessful polls the caller gets
// `false`, records kStatTimeout in the device status word and leaves through
// its normal exit path, so a lost copy can never hang the GPU.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "np_ring.h"

namespace npp {

constexpr int kStatTimeout = 8;           // a bounded wait ran out
constexpr uint32_t kSpinLimit = 1u << 20;  // polls; each poll may suspend for a short time

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// Makes barrier initialisation visible to the async (TMA) proxy.
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Orders this thread's earlier generic-proxy accesses to shared memory before
// later async-proxy (bulk copy) accesses.
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
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

// Bounded wait for the phase with the given parity to complete.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
  }
  return false;
}

// A bounded wait on an mbarrier for blocks that drain after a time-out: once any wait of the block has run out (*ok == 0)
// every later one of these is skipped.  True: the phase is complete.  One loop around one try_wait, not unrolled: with the unrolled
// loops of mbar_wait at every wait k_mlp_slices had 90 to 150 KB of code, missed the instruction cache on every layer (195
// times at 256 columns) and spent a sixth of its issue slots waiting for instructions.
__device__ __forceinline__ bool wait_or_flag(uint64_t* bar, uint32_t parity, volatile int* ok, int32_t* status) {
  uint32_t spin = 0;
#pragma unroll 1
  while (!mbar_try_wait(bar, parity)) {
    if (!*ok) return false;
    if (++spin == kSpinLimit) {
      *ok = 0;
      atomicOr(status, kStatTimeout);
    }
  }
  return true;
}

// A wait on a ring's own barriers, which the flag does not end (np_ring.h).  `ok` points to the flag and, behind it, to whether the
// ring was given up.  One sequence of the 7B shape takes 164.1 us per 32 layers with it, 162.3 with the wait above, which let the ring
// fall out of step; 13B 306.1 per 40 and 308.2.  (A producer that looks at the flag behind each wait for a free slot: 184.7.  Readers that
// give a slot back only while the flag stands: 163.8 and 312, eight sequences of the 13B shape 472 where this takes 468.)
struct RingBlock {
  volatile int* ok;
  int32_t* status;
  __device__ __forceinline__ bool stands() { return ok[0] != 0; }
  __device__ __forceinline__ void lower() {
    ok[0] = 0;
    atomicOr(status, kStatTimeout);
  }
  __device__ __forceinline__ void pause() { __nanosleep(4000); }
  __device__ __forceinline__ bool given_up() { return ok[1] != 0; }
  __device__ __forceinline__ void give_up() { ok[1] = 1; }
};
__device__ __forceinline__ void ring_wait(uint64_t* bar, uint32_t parity, volatile int* ok, int32_t* status) {
  RingBlock b = {ok, status};
  uint32_t polls = 0;
#pragma unroll 1
  while (!mbar_try_wait(bar, parity))
    if (ring_wait_step<kSpinLimit>(polls, b)) return;
}

// A block may leave only when the copies it has asked for have landed: after a time-out nobody else waits for them, and they
// would write to shared memory that is another block's by then.  `patience`: polls left to the block for all of this.
__device__ __forceinline__ void wait_landed(uint64_t* full, uint32_t parity, uint32_t& patience) {
#pragma unroll 1
  while (patience > 0 && !mbar_try_wait(full, parity)) --patience;
}
// For the one lane that fills a ring of `n` slots in turn, at its end: `next` is the slot it would fill next, in the use with
// parity `par`; the slots before it were filled in that use, the others in the one before (or never: the wait for a use before
// the first returns at once).
__device__ __forceinline__ void drain_ring(uint64_t* full, int n, int next, uint32_t par, uint32_t& patience) {
#pragma unroll 1
  for (int s = 0; s < n; ++s) wait_landed(&full[s], s < next ? par : par ^ 1u, patience);
}

// 1-D bulk copy global -> this CTA's shared memory; completion is reported to
// `bar` in bytes.  Both addresses 16-byte aligned, `bytes` a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst_smem, const void* src_gmem, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst_smem)),
      "l"(src_gmem), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Same, with an L2 evict-first policy: the data is read once.
__device__ __forceinline__ void bulk_g2s_stream(void* dst_smem, const void* src_gmem, uint32_t bytes,
                                                uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::
          "r"(smem_addr(dst_smem)),
      "l"(src_gmem), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
      : "memory");
}

__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// Programmatic dependent launch: let the next kernel in the stream start its
// prologue / wait until the previous kernel's memory is visible.
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait_prior() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace npp
