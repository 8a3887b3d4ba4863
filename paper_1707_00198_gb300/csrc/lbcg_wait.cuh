// Flags between the blocks of one cooperative grid (the resident step kernel, lbcg_run.cu, and the
// resident reverse sweep, lbcg_adjoint.cu): one word per block, counting upwards.
#pragma once

#include <cuda_runtime.h>

namespace lbcg {

__device__ __forceinline__ unsigned load_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void store_release(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Waits until the word at p has reached `want` (counts may wrap around).  Bounded: false after `limit`
// polls without it, or once another block has given up and set the error word (nothing of the
// caller's own is in flight then).
__device__ __forceinline__ bool wait_reached(const unsigned* p, unsigned want, int limit, const int* err) {
  for (int polls = 0; polls < limit; ++polls) {
    if (int(load_acquire(p) - want) >= 0) return true;
    if ((polls & 1023) == 1023 && *static_cast<const volatile int*>(err) != 0) return false;
  }
  return false;
}

}  // namespace lbcg
