// grid_sync.cuh -- grid-wide barrier of a cooperative launch, bounded in
// wall-clock time (the persistent kernels: the adjoint's segment kernels and
// the persistent form of the fused step).
#pragma once
#include <cstdint>

#include "tma.cuh"

namespace nlc {

// cumulative arrival counter, zeroed before each launch
struct GridBarrier {
  unsigned arrived;
};

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_gpu_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Grid-wide barrier of a cooperative launch, in two halves.  grid_arrive: thread
// 0 of each block adds its arrival with release semantics (the counter is
// cumulative: generation g completes at (g + 1) gridDim.x).  Returns, to thread
// 0, false where the wait is bounded by 0 ns and some other block has not
// arrived yet: such a wait runs out whatever the others do (the look comes
// before the block's own arrival, so that at least the first block of every
// generation gets false; looking afterwards, blocks that arrive within the
// round trip of one load all find the barrier complete).
__device__ __forceinline__ bool grid_arrive(GridBarrier* b, unsigned gen, uint64_t wait_ns) {
  __syncthreads();
  bool may_wait = true;
  if (threadIdx.x == 0) {
    if (wait_ns == 0) may_wait = ld_acquire_gpu(&b->arrived) + 1 >= (gen + 1) * gridDim.x;
    red_release_gpu_add(&b->arrived, 1u);
  }
  return may_wait;
}

// grid_wait: thread 0 polls the counter with acquire semantics until every block
// of this generation has arrived; work of the block that other blocks do not
// need can stand between the two halves.  The poll is bounded by wait_ns
// nanoseconds of %globaltimer; returns false in every thread of the block if
// it ran out.
__device__ __forceinline__ bool grid_wait(GridBarrier* b, unsigned& gen, unsigned* err,
                                          uint64_t wait_ns, bool may_wait) {
  int ok = 1;
  if (threadIdx.x == 0) {
    const unsigned target = (gen + 1) * gridDim.x;
    if (!may_wait) {
      ok = 0;
    } else if (ld_acquire_gpu(&b->arrived) < target) {
      const uint64_t t0 = global_ns();
      while (ok && ld_acquire_gpu(&b->arrived) < target)
        if (global_ns() - t0 >= wait_ns) ok = 0;
    }
    if (!ok) atomicExch(err, DEV_ERR_GRID_TIMEOUT);
  }
  gen++;
  return __syncthreads_and(ok) != 0;
}

__device__ __forceinline__ bool grid_sync(GridBarrier* b, unsigned& gen, unsigned* err,
                                          uint64_t wait_ns) {
  const bool may_wait = grid_arrive(b, gen, wait_ns);
  return grid_wait(b, gen, err, wait_ns, may_wait);
}

// orders this thread's earlier generic-proxy global writes (made visible
// by a grid barrier) before later async-proxy (TMA) reads of the same memory
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

}  // namespace nlc
