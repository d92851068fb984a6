// Shared-memory barrier, bulk-copy and tensor-core (tcgen05) primitives used
// by the kernels that stage their operands with asynchronous copies.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace feti {
namespace {

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t c) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(c) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t par) {
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok)
               : "r"(su32(b)), "r"(par)
               : "memory");
  return ok != 0;
}

// The same, held for hint_ns at most.
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t par, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok)
               : "r"(su32(b)), "r"(par), "r"(hint_ns)
               : "memory");
  return ok != 0;
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}

// Bounded wait: false after 2e8 SM clock cycles (about 0.1 s).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* b, uint32_t par) {
  const long long t0 = clock64();
  while (!mbar_try(b, par))
    if (clock64() - t0 > 200000000LL) return false;
  return true;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   su32(dst)),
               "l"(src), "r"(bytes), "r"(su32(b))
               : "memory");
}

// Shared-memory matrix descriptor: 128-byte swizzle, K-major, 1024 B between
// 8-row groups.
__device__ __forceinline__ uint64_t sw128_desc(const void* p) {
  uint64_t d = (su32(p) >> 4) & 0x3FFF;
  d |= (uint64_t)1 << 16;            // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;  // stride byte offset
  d |= (uint64_t)1 << 46;            // descriptor version
  d |= (uint64_t)2 << 61;            // 128-byte swizzle
  return d;
}

}  // namespace
}  // namespace feti
