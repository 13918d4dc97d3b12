// fma2.cuh -- two FP32 FMAs an instruction.
#pragma once

#include <cstdint>

namespace labsg {

// Two FP32 FMAs an instruction, each rounded as fmaf rounds: the FMA pipe's rate is the same, at half the issue
// slots, which the shared-memory loads and the packing of the operands then use.
__device__ __forceinline__ uint64_t pack2(float x, float y) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(x), "f"(y));
  return v;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ void ffma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

}  // namespace labsg
