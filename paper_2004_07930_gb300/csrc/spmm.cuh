// Sparse products on complex blocks [n][s], shared by the FP64 (kernels.cu),
// FP32 (krylov.cu) and double-float (df.cu) forms.
//
// Threads are (column, row) pairs; a row's index and value loads are shared by
// its s threads (one broadcast), and one nonzero reads one contiguous row of
// X. Narrow blocks (and small ones, which would not fill the SMs)
// give a row to T neighbouring lanes, which take every T-th nonzero and add
// their parts at the end.
//
// What bounds it, on the 5 Hz workload (0.95M rows, 43.7M nonzeros, 16 columns,
// double-float, 1.06 ms with the input's transpose, the output's columns
// written here; one thread per column and row, rows in their order, scalar
// arithmetic: 1.28): the FMA pipe's two cycles per
// packed instruction (0.45 ms) next to the latency of the X rows, half of
// which come from L2. DRAM has 0.8 GB to move, 0.12 ms.
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
struct SpF32 {  // ordered sums only
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
};
// Double-float values, the real and the imaginary part side by side in packed
// pairs (half the issue slots; the arithmetic of df_mac on each). X in
// double-float, (re hi, im hi, re lo, im lo) = two such pairs, or in FP32 (low
// parts zero: the same result as with them, one multiply-add less and half
// the bytes per entry).
template <typename XT>
struct SpDf {
  using Val = float2;
  using X = XT;
  struct Acc {
    pair2 h, l;
  };
  static __device__ __forceinline__ Acc zero() { return {pk(0.f, 0.f), pk(0.f, 0.f)}; }
  static __device__ __forceinline__ void mac(Acc& y, pair2 ah, pair2 na, pair2 al, float4 x) {
    df_mac2(y.h, y.l, ah, na, al, pk(x.x, x.y), pk(x.z, x.w));
  }
  static __device__ __forceinline__ void mac(Acc& y, pair2 ah, pair2 na, pair2 al, float2 x) {
    df_mac2(y.h, y.l, ah, na, al, pk(x.x, x.y));
  }
  static __device__ __forceinline__ float4 turn(float4 x) { return make_float4(x.y, x.x, x.w, x.z); }  // im, re
  static __device__ __forceinline__ float2 turn(float2 x) { return make_float2(x.y, x.x); }
  static __device__ __forceinline__ void re(Acc& y, Val a, X x) {
    mac(y, pk(a.x, a.x), pk(-a.x, -a.x), pk(a.y, a.y), x);
  }
  static __device__ __forceinline__ void im(Acc& y, Val b, X x) {  // re -= b im(x), im += b re(x)
    mac(y, pk(-b.x, b.x), pk(b.x, -b.x), pk(-b.y, b.y), turn(x));
  }
  static __device__ __forceinline__ Acc add(Acc a, Acc b) {
    df_add2(a.h, a.l, sub2(pk(0.f, 0.f), b.h), b.l);
    return a;
  }
  static __device__ __forceinline__ Acc shfl(Acc a, int off) {
    return {__shfl_down_sync(0xffffffffu, a.h, off), __shfl_down_sync(0xffffffffu, a.l, off)};
  }
  static __device__ __forceinline__ float4 parts(Acc a) {  // re hi, re lo, im hi, im lo
    const float2 h = unpk(a.h), l = unpk(a.l);
    return make_float4(h.x, l.x, h.y, l.y);
  }
  static __device__ __forceinline__ double2 to_d(Acc a) {
    const float4 p = parts(a);
    return make_double2(f2d(p.x) + f2d(p.y), f2d(p.z) + f2d(p.w));
  }
};

// y[i] += sum over a row's nonzeros p, p + T, ... < pe; Xc: the thread's first
// column, its second one dc entries on; pitch: bytes of a row of X
template <typename P, bool IM, int T, int CPT>
__device__ __forceinline__ void sp_row(typename P::Acc (&y)[CPT], int64_t p, int64_t pe,
                                       const int32_t* __restrict__ col, const typename P::Val* __restrict__ val,
                                       const typename P::X* __restrict__ Xc, int dc, uint32_t pitch) {
  const int32_t* cp = col + p;
  const typename P::Val* vp = val + p;
#pragma unroll 4
  for (int k = (int)(pe - p); k > 0; k -= T, cp += T, vp += T) {
    const typename P::Val a = __ldg(vp);
    const typename P::X* xp = reinterpret_cast<const typename P::X*>(reinterpret_cast<const char*>(Xc) +
                                                                     (uint64_t)(uint32_t)__ldg(cp) * pitch);
    typename P::X x[CPT];
#pragma unroll
    for (int i = 0; i < CPT; ++i) x[i] = __ldg(xp + i * dc);
#pragma unroll
    for (int i = 0; i < CPT; ++i)
      if (IM)
        P::im(y[i], a, x[i]);
      else
        P::re(y[i], a, x[i]);
  }
}

// From SP_LARGE entries on a block's rows are sorted within the CTA and, from
// SP_COL columns on, a thread takes two columns (FP32 and double-float; the
// FP64 pipe gains nothing from fewer loads and loses warps: 0.87 -> 1.04 ms on
// the quarter workload). Measured, 16 columns at 5 Hz: 1.28 ms, two columns
// 1.22, sorted 1.18, both 1.06; quarter, 5 columns, 1.2M entries: 0.206 ms
// with one column, 0.222 with two. Smaller blocks are bound by latency, which
// the sort's two barriers add to (quarter, 5 columns, coarse products of
// 180K entries: 5.95 -> 6.12 ms per two-level application).
constexpr int SP_COL = 16;
constexpr int64_t SP_LARGE = 400000;

// The CTA's rows in the order of their length, by runs of 32: threadIdx.y's
// row. Rows of the cubic space have 20 (a node of one boundary face) to 175
// nonzeros (a vertex), 45 on average, and a warp of two to
// ten rows works as long as its longest (25 of 32 lanes busy on average in
// their own order with two, 20 with four).
__device__ __forceinline__ int sp_rank(int64_t n, int s, const int64_t* __restrict__ rp) {
  __shared__ int len[256], ord[256];
  const int rows = blockDim.y, i = threadIdx.y * blockDim.x + threadIdx.x;
  if (n * s < SP_LARGE) return threadIdx.y;
  const int64_t r = blockIdx.x * (int64_t)rows + i;
  int l = -1;
  if (i < rows) {
    if (r < n) l = (int)(rp[r + 1] - rp[r]);
    len[i] = l;
  }
  __syncthreads();
  if (i < rows) {
    const int b = i & ~31, e = min(b + 32, rows);
    int k = b;
    for (int j = b; j < e; ++j) k += len[j] > l || (len[j] == l && j < i);
    ord[k] = i;
  }
  __syncthreads();
  return ord[threadIdx.y];
}

// out(row, column, sum) for every entry of (A_re + i A_im) X; rp_im NULL: A_re only.
// T lanes share a row, or a thread has CPT columns of it: c and c + blockDim.x.
// Registers for five or four CTAs per SM: with the compiler's own choice of 32
// the loads of four nonzeros did not stay in flight together (two-level, cube,
// 4 columns: 1.94 -> 1.71 ms per application).
template <typename P, int T, int CPT, typename Out>
__global__ void __launch_bounds__(256, CPT == 1 ? 5 : 4) k_spmm(int64_t n, int s, const int64_t* __restrict__ rp_re,
                                              const int32_t* __restrict__ col_re,
                                              const typename P::Val* __restrict__ val_re,
                                              const int64_t* __restrict__ rp_im, const int32_t* __restrict__ col_im,
                                              const typename P::Val* __restrict__ val_im,
                                              const typename P::X* __restrict__ X, Out out) {
  int64_t r;
  int c, t, dc = 0;
  if (T == 1) {  // block (columns / CPT, rows)
    r = blockIdx.x * (int64_t)blockDim.y + sp_rank(n, s, rp_re);
    c = blockIdx.y * (CPT * blockDim.x) + threadIdx.x;
    t = 0;
    if (r >= n || c >= s) return;
    if (CPT == 2 && c + (int)blockDim.x < s) dc = blockDim.x;  // else the first column twice
  } else {  // block (32, warps): 32 / (s T) rows per warp
    const int per = s * T, w = threadIdx.x / per, i = threadIdx.x - w * per;
    r = (blockIdx.x * (int64_t)blockDim.y + threadIdx.y) * (32 / per) + w;
    if (w >= 32 / per) r = n;
    t = i / s;
    c = i - t * s;
  }
  const uint32_t pitch = (uint32_t)s * sizeof(typename P::X);
  typename P::Acc y[CPT];
#pragma unroll
  for (int i = 0; i < CPT; ++i) y[i] = P::zero();
  if (r < n) {
    sp_row<P, false, T>(y, rp_re[r] + t, rp_re[r + 1], col_re, val_re, X + c, dc, pitch);
    if (rp_im) sp_row<P, true, T>(y, rp_im[r] + t, rp_im[r + 1], col_im, val_im, X + c, dc, pitch);
  }
  if constexpr (T > 1)
#pragma unroll
    for (int o = T / 2; o > 0; o /= 2) {
      const typename P::Acc z = P::shfl(y[0], o * s);
      if (t < o) y[0] = P::add(y[0], z);
    }
  if (r < n && t == 0) out(r, c, y[0]);
  if (CPT == 2 && dc > 0) out(r, c + dc, y[CPT - 1]);
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

template <typename P, int T, int CPT, typename Out>
void spmm_launch_t(int64_t n, int s, const int64_t* rp_re, const int32_t* col_re, const typename P::Val* val_re,
                   const int64_t* rp_im, const int32_t* col_im, const typename P::Val* val_im,
                   const typename P::X* X, Out out, cudaStream_t st) {
  // one lane per row: CTAs of one warp while there are not enough of eight warps for the SMs
  const int w = std::min((s + CPT - 1) / CPT, 256), threads = std::max(w, n * s < 80000 ? 32 : 256);
  const dim3 b = T == 1 ? dim3(w, threads / w) : dim3(32, 4);
  const int64_t rows = T == 1 ? b.y : (int64_t)b.y * (32 / (s * T));
  const dim3 g((unsigned)((n + rows - 1) / rows), T == 1 ? (s + CPT * w - 1) / (CPT * w) : 1);
  k_spmm<P, T, CPT, Out><<<g, b, 0, st>>>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out);
  count_launch();
}

// Lanes per row: as many as fit a warp, up to 8, while the block has fewer
// entries than the SMs have lanes to give them (cube of 6^3 cells, one column,
// FP64: 15 us with one lane, 6 with eight); on large blocks two to four where
// a row's s columns leave the index and value loads uncoalesced. ORDERED:
// one lane per row, every row summed in storage order (the operators of the
// inner coarse iteration, whose rounding the preconditioner amplifies).
template <typename P, bool ORDERED, typename Out>
void spmm_launch(int64_t n, int s, const int64_t* rp_re, const int32_t* col_re, const typename P::Val* val_re,
                 const int64_t* rp_im, const int32_t* col_im, const typename P::Val* val_im, const typename P::X* X,
                 Out out, cudaStream_t st) {
  if (n * s == 0) return;
  const bool small = n * s < 160000;
  if constexpr (ORDERED && std::is_same<P, SpF64>::value)
    if (small) {
      k_spmm_parts<<<(unsigned)((2 * n * s + 63) / 64), 64, 0, st>>>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im,
                                                                   reinterpret_cast<const double*>(X), out);
      count_launch();
      return;
    }
  if constexpr (!ORDERED) {
    const int fit = s <= 4 ? 8 : (s <= 8 ? 4 : (s <= 16 ? 2 : 1));
    const int T = small ? fit : (s <= 2 ? 4 : (s <= 4 ? 2 : 1));
    if (T == 8) return spmm_launch_t<P, 8, 1>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
    if (T == 4) return spmm_launch_t<P, 4, 1>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
    if (T == 2) return spmm_launch_t<P, 2, 1>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
  }
  if constexpr (!std::is_same<P, SpF64>::value)
    if (s >= SP_COL && n * s >= SP_LARGE)
      return spmm_launch_t<P, 1, 2>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
  spmm_launch_t<P, 1, 1>(n, s, rp_re, col_re, val_re, rp_im, col_im, val_im, X, out, st);
}

}  // namespace hz
