// Grid barrier of the resident step kernels (cooperative launches: every block of the grid is resident).
//
// An arrival counter in the context's memory that only grows; every wait is bounded (4 s of the GPU's
// global timer), and when one expires the block sets the context's error word and an abort word that ends
// every other wait, and all blocks return: the next pd_sync / pd_get_* reports PD_ERR_TIMEOUT.
#pragma once

#include "pd_internal.h"

namespace pd {
namespace {

struct GridBar {
  unsigned* bar;  // [0] arrivals, [1] abort
  unsigned base;  // arrivals before this launch
};

constexpr unsigned kPollLimit = 1u << 26;
constexpr unsigned long long kBarrierNs = 4000000000ull;  // other work on the GPU may hold a block back for a while

__device__ __forceinline__ unsigned ld_relaxed(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// All blocks of the grid: what any of them wrote before is visible to all of them after.  One thread of a
// block arrives with release and polls with acquire order, between two block barriers, so that the block's
// plain stores before and plain loads after are ordered too.  (A full fence on each side of the wait, and
// the timer read at its start, cost a step of a one-slice body 7.4 us where this takes 6.5 us.)  False
// when the wait expired or another block gave up.
__device__ __forceinline__ bool grid_barrier(const StepArgs& a, const GridBar& r, unsigned& target) {
  __shared__ int ok_s;
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    // testing (PD_OPT_EXPIRE_WAITS): block 0 never arrives
    if (!(a.expire && blockIdx.x == 0)) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(r.bar) : "memory");
    unsigned long long t0 = 0ull;
    for (unsigned it = 1; (int)(ld_acquire(r.bar) - target) < 0; ++it) {
      if ((it & 255u) != 0u) continue;
      const unsigned long long now = timer_ns();
      if (t0 == 0ull) t0 = now;
      if (ld_relaxed(r.bar + 1) != 0u || now - t0 > kBarrierNs || it > kPollLimit) {
        ok = 0;
        atomicExch(r.bar + 1, 1u);
        atomicExch(&a.counters[4], 1ull);
        break;
      }
    }
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

// The barrier's words, allocated and zeroed at the first resident launch of a build.
inline pd_status ensure_grid_bar(pd_ctx* c) {
  if (c->bar) return PD_OK;
  pd_status st = alloc(c, &c->bar, 2);
  if (st != PD_OK) return st;
  PD_CUDA(cudaMemsetAsync(c->bar, 0, 2 * sizeof(unsigned), c->stream));
  c->bar_base = 0;
  return PD_OK;
}

}  // namespace
}  // namespace pd
