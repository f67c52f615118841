// grid.cuh -- the grid-wide barrier and the thread numbering of the cooperative kernels (the sampled
// certificate and the final stage).  Nothing here is visible through the C ABI.
#pragma once

#include "common.cuh"

namespace bridges {

constexpr unsigned kSpinCap = 1u << 22;  // polls of a grid barrier before it gives up

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_add_release(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Grid-wide barrier for a cooperative launch, on a counter that only grows within the launch
// (cleared before it): barrier k ends once the counter reaches k * gridDim.  Thread 0 of each
// block counts its barriers in shared memory (*epoch), arrives with one release add that returns
// nothing, and polls the counter with acquire loads -- one round trip to memory per poll and
// none for the arrival (against about 3 us per barrier for an acquire-release add that returns,
// a generation word and its release store).  The block's writes are ordered before its thread 0
// by the block barrier, the release add publishes them, and the acquire that sees the count
// carries everyone's to the block.  Returns false if the wait gave up: the status word then holds
// BRIDGES_ETIMEDOUT (or an earlier error) and the caller must leave the kernel.  Every other
// block then gives up at its next barrier, so a block that would write a result after the last
// phase never gets there; *result (when not null) is set to that first error here instead, so
// that a caller never reads the result of an earlier call.
static __device__ __noinline__ bool grid_barrier(unsigned* bar_count, int32_t* status, int64_t* result, unsigned polls,
                                          unsigned* epoch) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    const unsigned target = (*epoch += 1) * gridDim.x;
    red_add_release(bar_count, 1u);
    if (!bounded_poll([&] { return (int)(ld_acquire(bar_count) - target) >= 0; }, polls)) {
      const int32_t first = atomicCAS(status, 0, BRIDGES_ETIMEDOUT_CODE);
      if (result) *result = (int64_t)(first != 0 ? first : BRIDGES_ETIMEDOUT_CODE);
      ok = 0;
    }
  }
  __syncthreads();
  return ok != 0;
}

// A test knob: the last block sleeps (a bounded time) before its first barrier, so that the others' wait
// there gives up.  Never set in normal use.
__device__ __forceinline__ void hold_last_block(int32_t hold_polls) {
  if (hold_polls > 0 && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0)
    for (int32_t i = 0; i < hold_polls; i++) __nanosleep(100);
}

__device__ __forceinline__ int64_t gtid() { return (int64_t)blockIdx.x * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int64_t gstride() { return (int64_t)gridDim.x * blockDim.x; }
// This thread's index among all threads with the warps dealt round-robin over the blocks (warp w
// of block b is global warp w * gridDim + b): a loop over fewer items than threads still spreads
// them over every SM, and each warp still takes 32 consecutive items.
__device__ __forceinline__ int64_t gspread() {
  return (((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) << 5) + (threadIdx.x & 31);
}

}  // namespace bridges
