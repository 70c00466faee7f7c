// Packed pairs of FP32 numbers (the f32x2 instructions of sm_100 and later).
// Each half of a pair takes exactly the IEEE operation that the scalar
// instruction of the same name would, so packing two independent scalar
// computations changes no bit of either; it halves the instructions issued.
#pragma once

#include <cuda_runtime.h>

namespace vfisv {

struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 f2_pack(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ f2 f2_dup(float x) { return f2_pack(x, x); }
__device__ __forceinline__ float f2_lo(f2 a) {
  return __uint_as_float(static_cast<unsigned>(a.v));
}
__device__ __forceinline__ float f2_hi(f2 a) {
  return __uint_as_float(static_cast<unsigned>(a.v >> 32));
}
// Both signs flipped (exact, not on the FMA pipe).
__device__ __forceinline__ f2 f2_neg(f2 a) { return f2_pack(-f2_lo(a), -f2_hi(a)); }
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}

}  // namespace vfisv
