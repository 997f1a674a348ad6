// Double-float ("float-float") arithmetic for the FP64 parts of the mixed
// form: the outer product with A (Eq. eq1) and the coarse product with E.
//
// GB300 issues 64 FP32 fused multiply-adds for every FP64 one, so an FP64
// product with A is bound by the FP64 pipe at any block width. Here a double
// is carried as an unevaluated sum hi + lo of two FP32 numbers (|lo| below
// one ulp of hi, about 47-48 significant bits), after Dekker (1971): the product
// of two such numbers keeps hi*hi exactly through one fused multiply-add
// (TwoProduct) plus the two cross terms, and every partial sum is added with
// Knuth's error-free TwoSum; the rounding errors of the low parts are summed
// in FP32. The relative error of a row sum of m terms is about m * 2^-48
// of sum |a_ij x_j| (FP64: m * 2^-53), far below what the residual test of
// FGMRES needs. All operations use the _rn intrinsics so that the compiler
// cannot contract a product and a sum into one FMA (which would break the
// error-free transformations). Magnitudes from about 2^-103 (1e-31) to 2^128
// keep the full precision; smaller ones are carried with FP32 precision, like
// the mixed form's FP32 local solves.
//
// Layouts: a complex FP64 block [n][s] double2 becomes [n][s] float4
// (re_hi, im_hi, re_lo, im_lo), 16 bytes per entry like the FP64 block, the
// operand pairs of the packed arithmetic; the
// real values of a split CSR matrix become float2 (hi, lo) per nonzero.
#include <cuda_runtime.h>

#include "df.cuh"
#include "kernels.cuh"
#include "spmm.cuh"

namespace hz {

namespace {
inline unsigned grid_for(int64_t work, int block) { return (unsigned)((work + block - 1) / block); }
}  // namespace

__global__ void k_to_df(const double2* __restrict__ X, float4* __restrict__ Y, int64_t count) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= count) return;
  const double2 x = X[g];
  const float2 r = df_split(x.x), i = df_split(x.y);
  Y[g] = make_float4(r.x, i.x, r.y, i.y);
}

namespace {
template <typename P>
struct OutRows {  // Y = A X, or B - A X
  double2* Y;
  const double2* B;
  int s;
  __device__ __forceinline__ void operator()(int64_t r, int c, typename P::Acc a) const {
    const int64_t g = r * s + c;
    const double2 y = P::to_d(a);
    if (B) {
      const double2 b = B[g];
      Y[g] = make_double2(b.x - y.x, b.y - y.y);
    } else {
      Y[g] = y;
    }
  }
};
template <typename P>
struct OutCols {  // Y = A X with the columns contiguous, [s][n]
  double2* Y;
  int64_t n;
  __device__ __forceinline__ void operator()(int64_t r, int c, typename P::Acc a) const {
    Y[(int64_t)c * n + r] = P::to_d(a);
  }
};
template <typename P>
struct OutDf {  // Y = A X in double-float, renormalised, (re hi, re lo, im hi, im lo)
  float4* Y;
  int s;
  __device__ __forceinline__ void operator()(int64_t r, int c, typename P::Acc a) const {
    float4 y = P::parts(a);
    df_norm(y.x, y.y);
    df_norm(y.z, y.w);
    Y[r * s + c] = y;
  }
};
template <bool ORDERED, typename XT, typename Out>
void spmm_df(const DevSplitCsr& A, const XT* X, Out out, int s, cudaStream_t st) {
  spmm_launch<SpDf<XT>, ORDERED>(A.n, s, A.rp_re, A.col_re, A.val_re_df, A.rp_im, A.col_im, A.val_im_df, X, out, st);
}
}  // namespace

void spmm_real_df(int64_t nrows, const int64_t* rp, const int32_t* col, const float2* val, const float4* X,
                  double2* Y, int s, cudaStream_t st) {
  spmm_launch<SpDf<float4>, true>(nrows, s, rp, col, val, nullptr, nullptr, nullptr, X,
                                  OutRows<SpDf<float4>>{Y, nullptr, s}, st);
}

void to_df(const double2* X, float4* Y, int64_t count, cudaStream_t st) {
  if (count) { k_to_df<<<grid_for(count, 256), 256, 0, st>>>(X, Y, count); count_launch(); }
}

void spmm_split_df(const DevSplitCsr& A, const float4* X, double2* Y, const double2* B, int s, cudaStream_t st) {
  if (B)  // t = v - A q feeds FP32 local solves: in storage order
    spmm_df<true>(A, X, OutRows<SpDf<float4>>{Y, B, s}, s, st);
  else
    spmm_df<false>(A, X, OutRows<SpDf<float4>>{Y, nullptr, s}, s, st);
}
void spmm_split_df_cols(const DevSplitCsr& A, const float4* X, double2* Y, int s, cudaStream_t st) {
  spmm_df<false>(A, X, OutCols<SpDf<float4>>{Y, A.n}, s, st);
}
void spmm_split_df(const DevSplitCsr& A, const float4* X, float4* Y, int s, cudaStream_t st) {
  spmm_df<false>(A, X, OutDf<SpDf<float4>>{Y, s}, s, st);
}
void spmm_split_df(const DevSplitCsr& A, const float2* X, double2* Y, int s, cudaStream_t st) {
  spmm_df<false>(A, X, OutRows<SpDf<float2>>{Y, nullptr, s}, s, st);
}
void spmm_split_df(const DevSplitCsr& A, const float2* X, float4* Y, int s, cudaStream_t st, bool ordered) {
  if (ordered)
    spmm_df<true>(A, X, OutDf<SpDf<float2>>{Y, s}, s, st);
  else
    spmm_df<false>(A, X, OutDf<SpDf<float2>>{Y, s}, s, st);
}

}  // namespace hz
