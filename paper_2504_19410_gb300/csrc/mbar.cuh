// mbarrier and bulk-copy helpers (inline PTX, sm_90 and later), with a
// bounded wait: no wait here can outlast its limit.
#pragma once
#include <cuda_runtime.h>

#include "fsa_consts.h"

namespace fsa {

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }
// orders this thread's earlier shared-memory accesses (generic proxy) before
// later bulk copies into the same memory (async proxy)
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// global -> shared, `bytes` a multiple of 16, both addresses 16-byte aligned
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// shared -> global bulk copy in this thread's bulk async group (`bytes` a
// multiple of 16, both addresses 16-byte aligned); commit closes the group;
// wait_read0 returns once the shared memory of every committed group has been
// read (it may be rewritten), wait0 once their writes are done.
__device__ __forceinline__ void bulk_s2g(void* dst, const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n" ::"l"(dst), "r"(smem_u32(src)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void bulk_wait0() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// true once the phase with this parity has completed; false after `limit`
// SM clock cycles
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity,
                                          long long limit = kWaitLimitCycles) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > limit) return false;
  }
  return true;
}


// Dynamic tiles: a kernel launched with one CTA per tile whose running CTAs
// take over tiles not started yet (clusterlaunchcontrol, sm_100 and later),
// so every SM keeps its full set of CTAs to the end.  (With a fixed share of
// tiles per CTA the scheduler's favoured CTAs finish early: a double-word
// middle pass ran at 23 of 32 resident warps on average.)  Thread 0 alone
// asks and reads the answers; `next` publishes them to the CTA.
struct TileQueue {
  uint4 resp;                // the answer to the request in flight
  unsigned long long bar;
  int next;                  // the next tile, -1 = none
  int pad;
};
static_assert(sizeof(TileQueue) == 32, "32 bytes of shared memory");
__device__ __forceinline__ void tile_request(TileQueue* q) {  // thread 0
  fence_proxy_async_smem();
  mbar_arrive_expect_tx(&q->bar, 16);
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];\n" ::"r"(
                   smem_u32(&q->resp)),
               "r"(smem_u32(&q->bar))
               : "memory");
}
// thread 0, before the CTA's first barrier: the first request
__device__ __forceinline__ void tile_queue_init(TileQueue* q) {
  mbar_init(&q->bar, 1);
  fence_mbar_init();
  q->next = -1;
  tile_request(q);
}
// The next tile of a CTA, -1 for none: wait() waits (bounded) for the answer
// and tells whether it came, read() decodes it, late() records a wait that gave
// up.  A tile that was granted is this CTA's alone, so the answer is taken
// however late it comes; only when a second wait gives up too are there no
// more tiles.
template <class Wait, class Read, class Late>
__host__ __device__ __forceinline__ int granted_tile(const Wait& wait, const Read& read, const Late& late) {
  if (!wait()) {
    late();
    if (!wait()) return -1;
  }
  return read();
}
// thread 0: the answer to the request in flight, published in `next` (read it
// after a barrier).  A wait that gives up is recorded in the fault word.
__device__ __forceinline__ void tile_answer(TileQueue* q, unsigned parity, unsigned int* fault) {
  q->next = granted_tile(
      [&] { return mbar_wait(&q->bar, parity); },
      [&]() -> int {
        unsigned ok, x;
        asm volatile(
            "{\n .reg .b128 r;\n .reg .pred p;\n ld.shared.b128 r, [%2];\n"
            " clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n selp.u32 %0, 1, 0, p;\n mov.u32 %1, 0;\n"
            " @p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, r;\n}\n"
            : "=r"(ok), "=r"(x)
            : "r"(smem_u32(&q->resp))
            : "memory");
        return ok ? (int)x : -1;
      },
      [&] {
        if (fault) atomicOr(fault, kWaitTimeout);
      });
}

}  // namespace fsa
