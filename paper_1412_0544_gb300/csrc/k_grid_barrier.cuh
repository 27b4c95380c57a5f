// k_grid_barrier.cuh -- what the persistent kernels share: the bounded-wait grid barrier and the
// loop over time blocks and items.
#pragma once
#include "rk4_internal.h"

namespace rk4d {

__device__ __forceinline__ long long global_ns() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid-wide barrier over the co-resident blocks of a cooperative launch.  Returns false when
// this block gave up waiting (or another block already did).
__device__ __forceinline__ bool grid_barrier(WsHeader *hdr, long long timeout_ns, int extra) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned *gen = &hdr->bar_gen;
    volatile int *status = &hdr->status;
    const unsigned g = *gen;
    __threadfence();
    const unsigned expected = gridDim.x + (unsigned)extra;
    const unsigned arrived = atomicAdd(&hdr->bar_count, 1u) + 1u;
    if (arrived == expected) {
      atomicExch(&hdr->bar_count, 0u);
      __threadfence();
      atomicAdd(&hdr->bar_gen, 1u);
    } else {
      const long long t0 = global_ns();
      while (*gen == g) {
        if ((*status & ST_TIMEOUT) || global_ns() - t0 > timeout_ns) {
          atomicOr(&hdr->status, ST_TIMEOUT);
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// The time blocks of a persistent launch: every resident block draws items until the time block's
// are gone, then all meet at the grid barrier.  item_fn(ki, in, out, cin, cout, item, K, G)
// processes one item and ends with a barrier of the block.
template <typename F> __device__ __forceinline__ void persistent_loop(const PersistentJob &job, F &&item_fn) {
  int64_t nblocks_t = job.cnt[0];
  for (int i = 1; i < job.nk; ++i) nblocks_t += job.cnt[i];
  int ki = 0;
  int64_t ki_end = job.cnt[0];  // the time block at which the next kval begins
  for (int64_t t = 0; t < nblocks_t; ++t) {
    while (t >= ki_end) ki_end += job.cnt[++ki];
    const int K = job.kval[ki];
    const int G = job.Gval[ki];
    const int64_t ntiles = job.ntiles[ki];
    const void *in = (t & 1) ? job.bufB : job.bufA;
    void *out = (t & 1) ? job.bufA : job.bufB;
    const void *cin = (t & 1) ? job.cB : job.cA;
    void *cout = (t & 1) ? job.cA : job.cB;
    // Items are handed out dynamically (an atomic counter per time-block parity), so blocks
    // that drew cheaper items take more and all reach the barrier together.  Block 0 clears
    // the other parity's counter for the next time block (the barrier orders it).
    unsigned long long *ctr = &job.hdr->work[t & 1];
    if (blockIdx.x == 0 && threadIdx.x == 0 && t > 0) job.hdr->work[(t + 1) & 1] = 0ull;
    __shared__ long long s_item;
    if (threadIdx.x == 0) s_item = (long long)atomicAdd(ctr, 1ull);
    __syncthreads();
    for (int64_t item = s_item; item < ntiles;) {
      item_fn(ki, in, out, cin, cout, item, K, G);
      // an item ends with a barrier, so every thread has read s_item before it is rewritten
      if (threadIdx.x == 0) s_item = (long long)atomicAdd(ctr, 1ull);
      __syncthreads();
      item = s_item;
    }
    if (t + 1 < nblocks_t || job.extra_arrivals > 0) {
      if (!grid_barrier(job.hdr, job.timeout_ns, job.extra_arrivals)) return;
    }
  }
}

}  // namespace rk4d
