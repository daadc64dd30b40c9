// hsga_sync.cuh -- what the bounded waits of the kernels share: relaxed 64-bit
// accesses to records in global memory, the GPU's global timer and the limit on
// polls.
#pragma once

#include <stdint.h>

namespace hsga {

constexpr uint32_t kMaxSpins = 1u << 22;  // polls of a record

__device__ __forceinline__ uint64_t ld_relaxed64(const uint64_t *p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_relaxed64(uint64_t *p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

}  // namespace hsga
