// Sparse products on complex blocks [n][s], shared by the FP64 (kernels.cu),
// FP32 (krylov.cu) and double-float (df.cu) forms.
//
// Threads are (column, row) pairs; a row's index and value loads are shared by
// its s threads (one broadcast), and one nonzero reads one contiguous row of
// X. Narrow blocks (and small ones, which would not fill the SMs)
// give a row to T neighbouring lanes, which take every T-th nonzero and add
// their parts at the end.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "kernels.cuh"

namespace hz {

// Operand sets: value, entry of X, accumulator.
struct SpF64 {
  using Val = double;
  using X = double2;
  using Acc = double2;
  static __device__ __forceinline__ Acc zero() { return make_double2(0.0, 0.0); }
  static __device__ __forceinline__ void re(Acc& y, Val a, X x) {  // y += a x
    y.x = fma(a, x.x, y.x);
    y.y = fma(a, x.y, y.y);
  }
  static __device__ __forceinline__ void im(Acc& y, Val b, X x) {  // y += i b x
    y.x = fma(-b, x.y, y.x);
    y.y = fma(b, x.x, y.y);
  }
  static __device__ __forceinline__ Acc add(Acc a, Acc b) { return make_double2(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ Acc shfl(Acc a, int off) {
    return make_double2(__shfl_down_sync(0xffffffffu, a.x, off), __shfl_down_sync(0xffffffffu, a.y, off));
  }
  static __device__ __forceinline__ double2 to_d(Acc a) { return a; }
};
struct SpF32 {
  using Val = float;
  using X = float2;
  using Acc = float2;
  static __device__ __forceinline__ Acc zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ void re(Acc& y, Val a, X x) {
    y.x = fmaf(a, x.x, y.x);
    y.y = fmaf(a, x.y, y.y);
  }
  static __device__ __forceinline__ void im(Acc& y, Val b, X x) {
    y.x = fmaf(-b, x.y, y.x);
    y.y = fmaf(b, x.x, y.y);
  }
  static __device__ __forceinline__ Acc add(Acc a, Acc b) { return make_float2(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ Acc shfl(Acc a, int off) {
    return make_float2(__shfl_down_sync(0xffffffffu, a.x, off), __shfl_down_sync(0xffffffffu, a.y, off));
  }
};
// double-float values; X in double-float, or in FP32 (low parts zero: the same
// result as the double-float entries (x, 0), with one multiply-add less and
// half the bytes per entry)
template <typename XT>
struct SpDf {
  using Val = float2;
  using X = XT;
  using Acc = float4;  // (re hi, re lo, im hi, im lo)
  static __device__ __forceinline__ Acc zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ void re(Acc& y, Val a, float4 x) {
    df_mac(y.x, y.y, a.x, a.y, x.x, x.y);
    df_mac(y.z, y.w, a.x, a.y, x.z, x.w);
  }
  static __device__ __forceinline__ void im(Acc& y, Val b, float4 x) {
    df_mac(y.x, y.y, -b.x, -b.y, x.z, x.w);  // re -= b im(x)
    df_mac(y.z, y.w, b.x, b.y, x.x, x.y);    // im += b re(x)
  }
  static __device__ __forceinline__ void re(Acc& y, Val a, float2 x) {
    df_mac_f(y.x, y.y, a.x, a.y, x.x);
    df_mac_f(y.z, y.w, a.x, a.y, x.y);
  }
  static __device__ __forceinline__ void im(Acc& y, Val b, float2 x) {
    df_mac_f(y.x, y.y, -b.x, -b.y, x.y);
    df_mac_f(y.z, y.w, b.x, b.y, x.x);
  }
  static __device__ __forceinline__ Acc add(Acc a, Acc b) {
    df_add(a.x, a.y, b.x, b.y);
    df_add(a.z, a.w, b.z, b.w);
    return a;
  }
  static __device__ __forceinline__ Acc shfl(Acc a, int off) {
    return make_float4(__shfl_down_sync(0xffffffffu, a.x, off), __shfl_down_sync(0xffffffffu, a.y, off),
                       __shfl_down_sync(0xffffffffu, a.z, off), __shfl_down_sync(0xffffffffu, a.w, off));
  }
  static __device__ __forceinline__ double2 to_d(Acc a) {
    return make_double2(f2d(a.x) + f2d(a.y), f2d(a.z) + f2d(a.w));
  }
};

// y += sum over a row's nonzeros p, p + T, ... < pe
template <typename P, bool IM, int T>
__device__ __forceinline__ void sp_row(typename P::Acc& y, int64_t p, int64_t pe, const int32_t* __restrict__ col,
                                       const typename P::Val* __restrict__ val, const typename P::X* __restrict__ Xc,
                                       int s) {
#pragma unroll 4
  for (; p < pe; p += T) {
    const typename P::Val a = __ldg(val + p);
    const typename P::X x = __ldg(Xc + (int64_t)__ldg(col + p) * s);
    if (IM)
      P::im(y, a, x);
    else
      P::re(y, a, x);
  }
}

// out(row, column, sum) for every entry of (A_re + i A_im) X; rp_im NULL: A_re only
template <typename P, int T, typename Out>
__global__ void __launch_bounds__(256) k_spmm(int64_t n, int s, const int64_t* __restrict__ rp_re,
                                              const int32_t* __restrict__ col_re,
                                              const typename P::Val* __restrict__ val_re,
                                              const int64_t* __restrict__ rp_im, const int32_t* __restrict__ col_im,
                                              const typename P::Val* __restrict__ val_im,
                                              const typename P::X* __restrict__ X, Out out) {
  int64_t r;
  int c, t;
  if (T == 1) {  // block (columns, rows)
    r = blockIdx.x * (int64_t)blockDim.y + threadIdx.y;
    c = blockIdx.y * blockDim.x + threadIdx.x;
    t = 0;
  } else {  // block (32, warps): 32 / (s T) rows per warp
    const int per = s * T, w = threadIdx.x / per, i = threadIdx.x - w * per;
    r = (blockIdx.x * (int64_t)blockDim.y + threadIdx.y) * (32 / per) + w;
    if (w >= 32 / per) r = n;
    t = i / s;
    c = i - t * s;
  }
  if (T == 1 && (r >= n || c >= s)) return;
  typename P::Acc y = P::zero();
  if (r < n) {
    sp_row<P, false, T>(y, rp_re[r] + t, rp_re[r + 1], col_re, val_re, X + c, s);
    if (rp_im) sp_row<P, true, T>(y, rp_im[r] + t, rp_im[r + 1], col_im, val_im, X + c, s);
  }
#pragma unroll
  for (int o = T / 2; o > 0; o /= 2) {
    const typename P::Acc z = P::shfl(y, o * s);
    if (t < o) y = P::add(y, z);
  }
  if (r < n && t == 0) out(r, c, y);
}

// FP64, one lane per row and component: small blocks summed in storage order.
// The real and the imaginary part are separate chains, and a warp's FP64
// multiply-add occupies its scheduler for 64 clocks, so that the two on two
// lanes halve the time of the longest row.
template <typename Out>
__global__ void __launch_bounds__(256) k_spmm_parts(int64_t n, int s, const int64_t* __restrict__ rp_re,
                                                    const int32_t* __restrict__ col_re,
                                                    const double* __restrict__ val_re,
                                                    const int64_t* __restrict__ rp_im,
                                                    const int32_t* __restrict__ col_im,
                                                    const double* __restrict__ val_im, const double* __restrict__ X,
                                                    Out out) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t r = g / (2 * s);
  const int i = (int)(g - r * (2 * s)), h = i & 1;
  double y = 0.0;
  if (r < n) {
#pragma unroll 8
    for (int64_t p = rp_re[r], pe = rp_re[r + 1]; p < pe; ++p)
      y = fma(__ldg(val_re + p), __ldg(X + (int64_t)__ldg(col_re + p) * (2 * s) + i), y);
    if (rp_im)
#pragma unroll 4
      for (int64_t p = rp_im[r], pe = rp_im[r + 1]; p < pe; ++p) {
        const double b = __ldg(val_im + p);
        y = fma(h ? b : -b, __ldg(X + (int64_t)__ldg(col_im + p) * (2 * s) + (i ^ 1)), y);
      }
  }
  const double z = __shfl_xor_sync(0xffffffffu, y, 1);
  if (r < n && h == 0) out(r, i >> 1, make_double2(y, z));
}

template <typename P, int T, typename Out>
void spmm_launch_t(int64_t n, int s, const int64_t* rp_re, const int32_t* col_re, const typename P::Val* val_re,
                   const int64_t* rp_im, const int32_t* col_im, const typename P::Val* val_im,
                   const typename P::X* X, Out out, cudaStream_t st) {
  // one lane per row: CTAs of one warp while there are not enough of eight warps for the SMs
  const int w = std::min(s, 256), threads = std::max(w, n * s < 80000 ? 32 : 256);
  const dim3 b = T == 1 ? dim3(w, threads / w) : dim3(32, 4);
  const int64_t rows = T == 1 ? b.y : (int64_t)b.y * (32 / (s * T));
  const dim3 g((unsigned)((n + rows - 1) / rows), T == 1 ? (s + w - 1) / w : 1);
  k_spmm<P, T, Out><<<g, b, 0, st>>>(n, s, rp_re, col_re, val_re, rp_im, col_im,
                                                                   val_im, X, out);
  count_launch();
}

// Lanes per row: as many as fit a warp, up to 8, while the block has fewer
// entries than the SMs have lanes to give them (cube of 6^3 cells, one column,
// FP64: 15 us with one lane, 6 with eight); on large blocks two to four where
// a row's s columns leave the index and value loads uncoalesced. `ordered`:
// one lane per row, every row summed in storage order (the operators of the
// inner coarse iteration, whose rounding the preconditioner amplifies).
template <typename P, typename Out>
void spmm_launch(int64_t n, int s, const int64_t* rp_re, const int32_t* col_re, const typename P::Val* val_re,
                 const int64_t* rp_im, const int32_t* col_im, const typename P::Val* val_im, const typename P::X* X,
                 Out out, cudaStream_t st, bool ordered = false) {
  if (n * s == 0) return;
  const bool small = n * s < 160000;
  if constexpr (std::is_same<P, SpF64>::value)
    if (ordered && small) {
      k_spmm_parts<<<(unsigned)((2 * n * s + 63) / 64), 64, 0, st>>>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im,
                                                                   reinterpret_cast<const double*>(X), out);
      count_launch();
      return;
    }
  const int fit = s <= 4 ? 8 : (s <= 8 ? 4 : (s <= 16 ? 2 : 1));
  const int T = ordered ? 1 : (small ? fit : (s <= 2 ? 4 : (s <= 4 ? 2 : 1)));
  if (T == 8)
    spmm_launch_t<P, 8>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
  else if (T == 4)
    spmm_launch_t<P, 4>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
  else if (T == 2)
    spmm_launch_t<P, 2>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
  else
    spmm_launch_t<P, 1>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
}

}  // namespace hz
