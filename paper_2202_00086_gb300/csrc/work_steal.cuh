// Work distribution of the plain FP64 and DF64 launches without a queue in
// memory: block index b stands for the rays [b chunk, (b + 1) chunk), and a
// running block whose rays are used up takes over the index of a block that
// has not started yet (Blackwell's cluster launch control, which cancels that
// block and returns its index). Every ray is traced once, by whichever block
// holds its index; nothing outlives the launch, and launches on other streams
// and graph replays have nothing in common.
//
// A plain launch with one ray per thread lasts as long as each warp's slowest
// ray, keeps a block resident until its last warp ends, and its last wave of
// blocks may be nearly empty. With stealing (against one ray per thread, ms):
//   FP64 render 400^2 42.2 -> 40.0, 800^2 112.6 -> 109.6; 640 x 320 Dormand-Prince
//   disk 49.6 -> 47.1; 400^2 q-metric 96.7 -> 90.1; 100,003 particles 7.9 -> 6.6;
//   DF64 render 800^2 35.3 -> 34.0; 600^2 disk 17.8 -> 17.3; 600,000 particles 11.3 -> 9.2.
// The MIXED kernels keep one ray per thread: dealing out rays through a queue
// in memory costs them 2-10 %.
// A request is answered in about a microsecond (20,000 blocks were dealt out
// this way in 18 us), and the next one is made ahead of need.
#pragma once

#include <cstdint>

#include "osiris_internal.h"

namespace osiris_impl {

// The block's rays [next, end) and its request; `lock` guards them. Each
// field is read and written by the lock's holder only.
struct StealPool {
  uint4 response;  // 16 bytes, written by the answer to a request
  unsigned long long barrier;
  unsigned long long next, end;
  unsigned phase;  // of the barrier
  int pending;     // 1: a request has not been answered yet
  unsigned lock;
};

__device__ __forceinline__ volatile StealPool& steal_pool() {
  __shared__ __align__(16) StealPool pool;
  return pool;
}

__device__ __forceinline__ unsigned shared_address(const volatile void* p) {
  return (unsigned)__cvta_generic_to_shared(const_cast<const void*>(p));
}

__device__ __forceinline__ void steal_set(const KernelArgs& A, unsigned index) {
  volatile StealPool& P = steal_pool();
  const unsigned long long begin = (unsigned long long)index * (unsigned long long)A.chunk;
  const unsigned long long end = begin + (unsigned long long)A.chunk;
  const unsigned long long total = (unsigned long long)A.total_rays;
  P.next = begin < total ? begin : total;
  P.end = end < total ? end : total;
}

// Ask for the index of a block that has not started.
__device__ __forceinline__ void steal_request() {
  volatile StealPool& P = steal_pool();
  const unsigned bar = shared_address(&P.barrier);
  // the answer to the previous request has been read before this one is written
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], 16;" ::"r"(bar) : "memory");
#ifndef OSIRIS_STEAL_MUTE  // test builds: no request is sent, so that no answer ever comes
  asm volatile(
      "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 "
      "[%0], [%1];" ::"r"(shared_address(&P.response)),
      "r"(bar)
      : "memory");
#endif
  P.pending = 1;
}

// All threads of the block, before any divergence.
__device__ __forceinline__ void steal_init(const KernelArgs& A) {
  volatile StealPool& P = steal_pool();
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(shared_address(&P.barrier))
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    P.phase = 0;
    P.lock = 0;
    steal_set(A, blockIdx.x);
    steal_request();
  }
  __syncthreads();
}

// Take the answer if it is there: a new index (and the next request), or none
// left (no request after that). Called by the lock's holder.
__device__ __forceinline__ void steal_answer(const KernelArgs& A) {
  volatile StealPool& P = steal_pool();
  unsigned there;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(there)
      : "r"(shared_address(&P.barrier)), "r"(P.phase)
      : "memory");
  if (!there) return;
  unsigned taken, index;
  asm volatile(
      "{\n\t.reg .b128 a;\n\t.reg .pred p;\n\t"
      "ld.shared.b128 a, [%2];\n\t"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, a;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t"
      "mov.u32 %1, 0;\n\t"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, a;\n\t}"
      : "=r"(taken), "=r"(index)
      : "r"(shared_address(&P.response))
      : "memory");
  P.phase ^= 1;
  P.pending = 0;
  if (taken) {
    steal_set(A, index);
    steal_request();
  }
}

// One ray for each lane of the warp that needs one, under the rule of
// refill() (trace_kernel.cuh). Returns 1 with the lane's ray in `first`, or 0;
// `over` (the same in every lane) when the block will get no more rays.
// Never waits: a lock that another warp holds, or an answer that is not there
// yet, leaves the lane idle until it asks again.
__device__ __forceinline__ int steal_refill(const KernelArgs& A, bool need, bool busy,
                                            int64_t& first, bool& over) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned m = __ballot_sync(FULL, need);
  const unsigned b = __ballot_sync(FULL, busy);
  over = false;
  if (!m || (b && __popc(m) < A.refill_lanes)) return 0;
  const int leader = __ffs(m) - 1;
  unsigned long long base = 0;
  unsigned got = 0;
  if (lane == leader) {
    volatile StealPool& P = steal_pool();
    unsigned* lock = const_cast<unsigned*>(&P.lock);
    if (atomicCAS(lock, 0u, 1u) == 0u) {
      __threadfence_block();
      if (P.next == P.end && P.pending) steal_answer(A);
      base = P.next;
      const unsigned long long left = P.end - base;
      const unsigned want = __popc(m);
      got = left < want ? (unsigned)left : want;
      P.next = base + got;
      if (got == 0 && !P.pending) got = 0x80000000u;  // over
      __threadfence_block();
      atomicExch(lock, 0u);
    }
  }
  base = __shfl_sync(FULL, base, leader);
  got = __shfl_sync(FULL, got, leader);
  if (got & 0x80000000u) {
    over = true;
    return 0;
  }
  const unsigned rank = __popc(m & ((1u << lane) - 1u));
  if (!need || rank >= got) return 0;
  first = (int64_t)(base + rank);
  return 1;
}

// Turns in a row that a warp without any ray waits for more of them. It waits
// only while the block's request is unanswered, about a microsecond, and a turn
// takes some hundred cycles, so 2^24 of them are a second or more. (A count of
// turns, not a time: it stands still while the GPU runs something else.)
#ifndef OSIRIS_STEAL_PATIENCE
#define OSIRIS_STEAL_PATIENCE (1u << 24)
#endif
constexpr unsigned kStealPatience = OSIRIS_STEAL_PATIENCE;

// Whether a warp without any ray asks again. It leaves once the block gets no
// more rays (`drained`), with no request outstanding then, or when its wait has
// run out. That is counted in the stats, and the rays that such a block may
// have taken over and not traced keep the OSIRIS_STATUS_NONE that the launch
// starts with.
__device__ __forceinline__ bool steal_waits(const KernelArgs& A, bool drained, unsigned& turns) {
  if (drained) return false;
  if (++turns <= kStealPatience) return true;
  if ((threadIdx.x & 31) == 0 && A.stats) atomicAdd(A.stats + OSIRIS_STAT_GAVE_UP, 1ull);
  return false;
}

}  // namespace osiris_impl
