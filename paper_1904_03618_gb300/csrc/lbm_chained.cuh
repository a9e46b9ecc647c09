// Waiting and loading in kernels launched with programmatic stream
// serialisation (the box form of the step, the surrogate's training step).
#pragma once

#include <cuda_runtime.h>
#include <string.h>

namespace lbm {

// Kernels launched with programmatic stream serialisation start while the one
// before them still runs.  after_previous_kernel returns once that one has
// completed and its stores are visible; only then may the next one start, so
// that at most two kernels of a chain are on the GPU at once.
__device__ __forceinline__ void after_previous_kernel() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
// Their loads of what earlier kernels of the chain write, ordered behind the
// wait.  Not __ldg (nor const __restrict__): the read-only path is for data that
// nobody writes while the kernel is on the GPU, waiting included.
__device__ __forceinline__ float ld_chained(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];\n" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_chained(const float2* p) {
  float2 v;
  asm volatile("ld.global.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_chained(const float4* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
template <typename Pair16>  // __half2, __nv_bfloat162
__device__ __forceinline__ Pair16 ld_chained(const Pair16* p) {
  static_assert(sizeof(Pair16) == 4, "a pair of 16-bit values");
  unsigned r;
  asm volatile("ld.global.b32 %0, [%1];\n" : "=r"(r) : "l"(p) : "memory");
  Pair16 v;
  memcpy(&v, &r, 4);
  return v;
}

}  // namespace lbm
