// grid_barrier.cuh -- a barrier over the blocks of a cooperative launch.
#pragma once

#include "common.cuh"

namespace mc {

constexpr unsigned kGridAbort = ~0u;

struct GridBar {  // zeroed before the launch
  unsigned arrived;
  unsigned pad[31];
  unsigned release;  // the last barrier complete, or kGridAbort
  unsigned pad2[31];
};

// Grid barrier number `gen` (1, 2, ...): false when the wait ran out (here or
// in another block; the error is set), after which every block leaves.  The last block to arrive
// releases the others through a word of its own line: the arrivals, atomics on
// one word, do not queue up behind the polls (with both on one word a barrier
// of 608 blocks took ~10 us).
__device__ __forceinline__ bool grid_barrier(GridBar* c, unsigned gen, long long spin, int* s_ok,
                                           DevState* st) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    bool ok = true;
    if (atomicAdd(&c->arrived, 1u) + 1u == gen * gridDim.x) {
      asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&c->release), "r"(gen) : "memory");
    } else {
      unsigned v = 0;
      long long it = 0;
      for (;;) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&c->release) : "memory");
        if (v >= gen) break;
        if (++it > spin) {  // (the value ends the wait of the others, too)
          asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&c->release), "r"(kGridAbort)
                       : "memory");
          set_error(st, ERR_TIMEOUT);
          v = kGridAbort;
          break;
        }
        __nanosleep(20);
      }
      ok = v != kGridAbort;
    }
    __threadfence();
    *s_ok = ok ? 1 : 0;
  }
  __syncthreads();
  return *s_ok != 0;
}

}  // namespace mc
