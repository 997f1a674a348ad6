// Packed FP32 arithmetic, shared by the front sweeps (sweep.cu) and the
// double-float products (spmm.cuh).
#pragma once
#include <cuda_runtime.h>

namespace hz {

// Packed pairs of FP32 numbers: the .f32x2 instructions round each half like
// the scalar ones, and issue half as many.
using pair2 = unsigned long long;
static __device__ __forceinline__ pair2 pk(float a, float b) {
  pair2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
static __device__ __forceinline__ float2 unpk(pair2 p) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(p));
  return r;
}
static __device__ __forceinline__ pair2 fma2(pair2 a, pair2 b, pair2 c) {
  pair2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
static __device__ __forceinline__ pair2 mul2(pair2 a, pair2 b) {
  pair2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
static __device__ __forceinline__ pair2 add2(pair2 a, pair2 b) {
  pair2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
static __device__ __forceinline__ pair2 sub2(pair2 a, pair2 b) {
  pair2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

}  // namespace hz
