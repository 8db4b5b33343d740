// Helpers shared by the two selection kernels (select.cu: one CTA per (sequence, head);
// select_cluster.cu: a thread-block cluster per (sequence, head)).
#pragma once

namespace cc {

// Order-preserving map from f32 to u32 (larger float <=> larger key); -0.0 ranks equal to +0.0.
__device__ __forceinline__ unsigned mono_key(float x) {
  unsigned b = __float_as_uint(__fadd_rn(x, 0.0f));
  return b ^ ((unsigned)((int)b >> 31) | 0x80000000u);
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// The float of a key (+0.0 for both zeros).
__device__ __forceinline__ float mono_value(unsigned key) {
  return __uint_as_float(key ^ (~(unsigned)((int)key >> 31) | 0x80000000u));
}

__device__ __forceinline__ unsigned warp_sum(unsigned v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace cc
