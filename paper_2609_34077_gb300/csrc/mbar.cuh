// Shared-memory mbarriers (sm_90+ PTX) of the tensor-core expert GEMMs; their bounded waits are in
// tc_ptx.cuh. Not part of the C ABI.
#pragma once

#include "common.cuh"

namespace mcft {

// Limit of every bounded mbarrier wait: after it the waiter records MCFT_ERR_TIMEOUT and returns.
constexpr uint64_t kTimeoutNs = 2000000000ull;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
}  // namespace mcft
