// Device helpers shared by the fp32 CUDA-core kernels: asynchronous 16-byte copies to shared
// memory and the row stride of its tiles.
#pragma once
#include <cstdint>

namespace moa {
namespace f32 {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// 16 bytes global -> shared, asynchronous.
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  const size_t g = __cvta_generic_to_global(src);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Shared-memory row stride, in floats, of a tile whose rows are read 16 bytes at a time by lanes
// that hold different rows: an odd number of 16-byte units, so 8 consecutive rows fall on
// disjoint banks.
__host__ __device__ constexpr int odd_stride(int d) { return ((d / 4) | 1) * 4; }

}  // namespace f32
}  // namespace moa
