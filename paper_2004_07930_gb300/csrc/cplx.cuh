// Complex helpers shared by the front sweeps (sweep.cu, mf.cu), on double2
// or float2.
#pragma once
#include <cuda_runtime.h>

namespace hz {

static __device__ __forceinline__ double2 mk2(double a, double b) { return make_double2(a, b); }
static __device__ __forceinline__ float2 mk2(float a, float b) { return make_float2(a, b); }

template <typename V>
static __device__ __forceinline__ V c_zero() {
  return mk2((decltype(V::x))0, (decltype(V::x))0);
}
template <typename V>
static __device__ __forceinline__ V c_fma(V a, V b, V c) {  // a*b + c
  return mk2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
template <typename V>
static __device__ __forceinline__ V c_mul(V a, V b) {
  return mk2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename V>
static __device__ __forceinline__ V c_add(V a, V b) {
  return mk2(a.x + b.x, a.y + b.y);
}

// Programmatic dependent launch (sm_90 and later): a kernel launched with
// programmatic stream serialisation may start while its predecessor in the
// stream is finishing; pdl_wait() blocks until the predecessor has completed
// and its writes are visible, pdl_trigger() lets the successor be scheduled.
// Both are no-ops for kernels launched without the attribute.
static __device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
static __device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch with programmatic stream serialisation when `pdl` (the front
// sweeps' launches: the next level's CTAs are scheduled while the previous
// launch drains and read their factors before pdl_wait()).
template <typename... P, typename... A>
static void launch_k(bool pdl, void (*k)(P...), unsigned grid, unsigned block, size_t shm, cudaStream_t st,
                     A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = shm;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, std::forward<A>(args)...);
  count_launch();
}

}  // namespace hz
