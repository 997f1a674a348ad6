// Device kernels of the two-level ORAS preconditioned FGMRES iteration.
//
// Sec. "Domain decomposition preconditioner": each GMRES iteration applies
// A (Eq. eq1) and M^{-1} (Eq. 2lvl): a coarse restriction Z^T, the coarse
// solve, the prolongation Z, a residual with A, the restriction R_i to every
// overlapping subdomain, the local solves A_i^{-1} (multifrontal LDL^T
// factors here, the paper's direct local solver) and the partition-of-unity
// prolongation sum_i R_i^T D_i (Eq. oras). Blocks of right-hand sides are
// stored row-major [n][s] (the s columns of a row contiguous), complex128 as
// double2 (re, im).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>

#include "kernels.cuh"
#include "spmm.cuh"

namespace hz {

std::atomic<long long> g_kernel_launches{0};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 c) {  // a*b + c
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
__device__ __forceinline__ double2 cfms(double2 a, double2 b, double2 c) {  // c - a*b
  return make_double2(fma(-a.x, b.x, fma(a.y, b.y, c.x)), fma(-a.x, b.y, fma(-a.y, b.x, c.y)));
}
__device__ __forceinline__ double2 conjmul_acc(double2 a, double2 b, double2 c) {  // conj(a)*b + c
  return make_double2(fma(a.x, b.x, fma(a.y, b.y, c.x)), fma(a.x, b.y, fma(-a.y, b.x, c.y)));
}
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double cabs2(double2 a) { return a.x * a.x + a.y * a.y; }

static inline unsigned grid_for(int64_t work, int block) { return (unsigned)((work + block - 1) / block); }

// ---------------------------------------------------------------------------
// SpMM: Y = (A_re + i A_im) X  or  Y = B - A X   (K1), native FP64
// ---------------------------------------------------------------------------
namespace {
struct OutRows {
  double2* Y;
  const double2* B;
  int s;
  __device__ __forceinline__ void operator()(int64_t r, int c, double2 y) const {
    const int64_t g = r * s + c;
    if (B) {
      const double2 b = B[g];
      y = make_double2(b.x - y.x, b.y - y.y);
    }
    Y[g] = y;
  }
};
struct OutCols {  // Y = A X with the columns contiguous, [s][n]
  double2* Y;
  int64_t n;
  __device__ __forceinline__ void operator()(int64_t r, int c, double2 y) const { Y[(int64_t)c * n + r] = y; }
};
}  // namespace

void spmm_split(const DevSplitCsr& A, const double2* X, double2* Y, const double2* B, int s, cudaStream_t st,
                bool ordered) {
  if (ordered)
    spmm_launch<SpF64, true>(A.n, s, A.rp_re, A.col_re, A.val_re, A.rp_im, A.col_im, A.val_im, X, OutRows{Y, B, s}, st);
  else
    spmm_launch<SpF64, false>(A.n, s, A.rp_re, A.col_re, A.val_re, A.rp_im, A.col_im, A.val_im, X, OutRows{Y, B, s}, st);
}
void spmm_split_cols(const DevSplitCsr& A, const double2* X, double2* Y, int s, cudaStream_t st) {
  spmm_launch<SpF64, false>(A.n, s, A.rp_re, A.col_re, A.val_re, A.rp_im, A.col_im, A.val_im, X, OutCols{Y, A.n}, st);
}

void spmm_real(int64_t nrows, const int64_t* rp, const int32_t* col, const double* val, const double2* X,
               double2* Y, int s, cudaStream_t st) {
  spmm_launch<SpF64, true>(nrows, s, rp, col, val, nullptr, nullptr, nullptr, X, OutRows{Y, nullptr, s}, st);
}

// ---------------------------------------------------------------------------
// Restriction R_i (gather, K2) and Boolean partition-of-unity prolongation
// sum_i R_i^T D_i (each dof read from its owning subdomain copy, K3)
// ---------------------------------------------------------------------------
// Threads are (column, row) pairs, so that no index is divided by the block
// width; a sub-vector row has `cols` entries, those from s on zero.
template <typename In, typename Out>
__global__ void k_gather(const int* __restrict__ idx, int64_t nrows, const In* __restrict__ X, Out* __restrict__ Y, int s,
                         int cols) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.y + threadIdx.y;
  const int c = threadIdx.x;
  if (r >= nrows) return;
  Out y;
  y.x = y.y = 0;
  if (c < s) {
    const In x = X[(int64_t)idx[r] * s + c];
    y.x = (decltype(y.x))x.x;
    y.y = (decltype(y.y))x.y;
  }
  Y[r * cols + c] = y;
}

// the operand of the product that follows: z in double-float, or in FP32 where z has no more
__device__ __forceinline__ void put_copy(float4* p, double2 z) {
  const float2 a = df_split(z.x), b = df_split(z.y);
  *p = make_float4(a.x, b.x, a.y, b.y);
}
__device__ __forceinline__ void put_copy(float4* p, float2 z) { *p = make_float4(z.x, z.y, 0.f, 0.f); }

template <typename In, typename Q, typename Out>
__global__ void k_scatter(const int* __restrict__ own, int64_t n, const In* __restrict__ Xsub, const Q* __restrict__ Qb,
                          Out* __restrict__ Z, int s, int cols, float4* __restrict__ Zdf, float2* __restrict__ Zf) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.y + threadIdx.y;
  const int c = threadIdx.x;
  if (r >= n) return;
  const In x = Xsub[(int64_t)own[r] * cols + c];
  Out z;
  z.x = x.x;
  z.y = x.y;
  if (Qb) {
    const Q q = Qb[r * s + c];
    z.x += (decltype(z.x))q.x;
    z.y += (decltype(z.y))q.y;
  }
  Z[r * s + c] = z;
  if (Zdf) put_copy(Zdf + r * s + c, z);
  if (Zf) Zf[r * s + c] = make_float2((float)x.x, (float)x.y);
}

template <typename In, typename Out>
static void gather_t(const DevMF& mf, const In* X, Out* Y, int s, cudaStream_t st) {
  const int64_t nrows = mf.nsub_rows;
  if (nrows * s == 0) return;
  const int cols = sub_cols(mf, s);
  const dim3 b(cols, std::max(1, 256 / cols));
  { k_gather<<<grid_for(nrows, b.y), b, 0, st>>>(mf.gidx, nrows, X, Y, s, cols); count_launch(); }
}
template <typename In, typename Q, typename Out>
static void scatter_t(const DevMF& mf, int64_t n, const In* Xsub, const Q* Qb, Out* Z, int s, cudaStream_t st,
                      float4* Zdf = nullptr, float2* Zf = nullptr) {
  if (n * s == 0) return;
  const dim3 b(s, std::max(1, 256 / s));
  { k_scatter<<<grid_for(n, b.y), b, 0, st>>>(mf.own, n, Xsub, Qb, Z, s, sub_cols(mf, s), Zdf, Zf); count_launch(); }
}

void gather_rows(const DevMF& mf, const double2* X, double2* Y, int s, cudaStream_t st) {
  gather_t(mf, X, Y, s, st);
}
void gather_rows(const DevMF& mf, const double2* X, float2* Y, int s, cudaStream_t st) {
  gather_t(mf, X, Y, s, st);
}
void gather_rows(const DevMF& mf, const float2* X, float2* Y, int s, cudaStream_t st) {
  gather_t(mf, X, Y, s, st);
}
void scatter_owned(const DevMF& mf, int64_t n, const double2* Xsub, const double2* Q, double2* Z, int s,
                   cudaStream_t st) {
  scatter_t(mf, n, Xsub, Q, Z, s, st);
}
void scatter_owned(const DevMF& mf, int64_t n, const float2* Xsub, const double2* Q, double2* Z, int s,
                   cudaStream_t st, float4* Zdf, float2* Zf) {
  scatter_t(mf, n, Xsub, Q, Z, s, st, Zdf, Zf);
}
void scatter_owned(const DevMF& mf, int64_t n, const float2* Xsub, const float2* Q, double2* Z, int s,
                   cudaStream_t st, float4* Zdf) {
  scatter_t(mf, n, Xsub, Q, Z, s, st, Zdf);
}
void scatter_owned(const DevMF& mf, int64_t n, const float2* Xsub, const float2* Q, float2* Z, int s, cudaStream_t st) {
  scatter_t(mf, n, Xsub, Q, Z, s, st);
}

__global__ void k_zero(double2* X, int64_t count) {
  int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g < count) X[g] = make_double2(0.0, 0.0);
}
void axpy_cols_zero(double2* X, int64_t count, cudaStream_t st) {
  if (count) { k_zero<<<grid_for(count, 256), 256, 0, st>>>(X, count); count_launch(); }
}

// one column c of an [n][s] block: zero it, copy it to another block, or
// extract it as a contiguous vector
__global__ void k_col_zero(double2* X, int64_t n, int s, int c) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) X[i * s + c] = make_double2(0.0, 0.0);
}
__global__ void k_col_copy(const double2* __restrict__ X, double2* __restrict__ Y, int64_t n, int s, int c) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) Y[i * s + c] = X[i * s + c];
}
__global__ void k_col_get(const double2* __restrict__ X, double2* __restrict__ y, int64_t n, int s, int c) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) y[i] = X[i * s + c];
}
void col_zero(double2* X, int64_t n, int s, int c, cudaStream_t st) {
  if (n) { k_col_zero<<<grid_for(n, 256), 256, 0, st>>>(X, n, s, c); count_launch(); }
}
void col_copy(const double2* X, double2* Y, int64_t n, int s, int c, cudaStream_t st) {
  if (n) { k_col_copy<<<grid_for(n, 256), 256, 0, st>>>(X, Y, n, s, c); count_launch(); }
}
void col_get(const double2* X, double2* y, int64_t n, int s, int c, cudaStream_t st) {
  if (n) { k_col_get<<<grid_for(n, 256), 256, 0, st>>>(X, y, n, s, c); count_launch(); }
}

// ---------------------------------------------------------------------------
// Right-hand sides (K11) and layout changes
// ---------------------------------------------------------------------------
__global__ void k_point_sources(double2* B, const int* __restrict__ idx, const double2* __restrict__ val, int nent) {
  int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < nent) B[idx[e]] = cadd(B[idx[e]], val[e]);
}
void scatter_point_sources(double2* B, int64_t n, int s, const int* idx, const double2* val, int nent,
                           cudaStream_t st) {
  (void)n;
  (void)s;
  if (nent) { k_point_sources<<<grid_for(nent, 128), 128, 0, st>>>(B, idx, val, nent); count_launch(); }
}

// [s][n] <-> [n][s], through a tile of TR rows and up to TCOL columns
// (blockIdx.y) so that both sides are read and written in full lines; to_rows
// also in double-float (the operand of the product, without the FP64 rows in
// between)
constexpr int TR = 32, TCOL = 64;
__device__ __forceinline__ void put_row(double2* p, double2 v) { *p = v; }
__device__ __forceinline__ void put_row(float4* p, double2 v) { put_copy(p, v); }
template <typename Out>
__global__ void __launch_bounds__(256) k_to_rows(const double2* __restrict__ F, Out* __restrict__ B, int64_t n, int s) {
  extern __shared__ double2 tile[];  // [columns][TR + 1]
  const int64_t r0 = blockIdx.x * (int64_t)TR;
  const int nr = (int)min((int64_t)TR, n - r0), c0 = blockIdx.y * TCOL, nc = min(TCOL, s - c0);
  for (int e = threadIdx.x; e < TR * nc; e += blockDim.x) {
    const int c = e / TR, r = e % TR;
    if (r < nr) tile[c * (TR + 1) + r] = F[(int64_t)(c0 + c) * n + r0 + r];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nr * nc; e += blockDim.x) {
    const int r = e / nc, c = e - r * nc;
    put_row(B + (r0 + r) * s + c0 + c, tile[c * (TR + 1) + r]);
  }
}
__global__ void __launch_bounds__(256) k_from_rows(const double2* __restrict__ B, double2* __restrict__ F, int64_t n,
                                                   int s) {
  extern __shared__ double2 tile[];
  const int64_t r0 = blockIdx.x * (int64_t)TR;
  const int nr = (int)min((int64_t)TR, n - r0), c0 = blockIdx.y * TCOL, nc = min(TCOL, s - c0);
  for (int e = threadIdx.x; e < nr * nc; e += blockDim.x) {
    const int r = e / nc, c = e - r * nc;
    tile[c * (TR + 1) + r] = B[(r0 + r) * s + c0 + c];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < TR * nc; e += blockDim.x) {
    const int c = e / TR, r = e % TR;
    if (r < nr) F[(int64_t)(c0 + c) * n + r0 + r] = tile[c * (TR + 1) + r];
  }
}
// one column: the two layouts are the same
__global__ void k_copy(const double2* __restrict__ X, double2* __restrict__ Y, int64_t count) {
  int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g < count) Y[g] = X[g];
}
static dim3 tile_grid(int64_t n, int s) { return dim3(grid_for(n, TR), (s + TCOL - 1) / TCOL); }
static size_t tile_bytes(int s) { return (size_t)std::min(s, TCOL) * (TR + 1) * sizeof(double2); }  // at most 33 KB
void transpose_to_rows(const double2* F, double2* B, int64_t n, int s, cudaStream_t st) {
  if (n * s == 0) return;
  if (s == 1) return cast_copy(F, B, n, st);
  { k_to_rows<<<tile_grid(n, s), 256, tile_bytes(s), st>>>(F, B, n, s); count_launch(); }
}
void transpose_to_rows(const double2* F, float4* B, int64_t n, int s, cudaStream_t st) {
  if (n * s == 0) return;
  if (s == 1) return to_df(F, B, n, st);
  { k_to_rows<<<tile_grid(n, s), 256, tile_bytes(s), st>>>(F, B, n, s); count_launch(); }
}
void transpose_from_rows(const double2* B, double2* F, int64_t n, int s, cudaStream_t st) {
  if (n * s == 0) return;
  if (s == 1) return cast_copy(B, F, n, st);
  { k_from_rows<<<tile_grid(n, s), 256, tile_bytes(s), st>>>(B, F, n, s); count_launch(); }
}

// debug_bounds: every entry a[i * stride] must lie in [lo, hi); the smallest
// failing check id is kept in *err (initialised to INT_MAX by the caller)
__global__ void k_check_range(const int* __restrict__ a, int64_t count, int stride, int64_t lo, int64_t hi,
                              int* __restrict__ err, int id) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int64_t v = a[i * stride];
  if (v < lo || v >= hi) atomicMin(err, id);
}
void check_index_range(const int* a, int64_t count, int stride, int64_t lo, int64_t hi, int* err, int id,
                       cudaStream_t st) {
  if (count > 0 && a) { k_check_range<<<grid_for(count, 256), 256, 0, st>>>(a, count, stride, lo, hi, err, id); count_launch(); }
}

void cast_copy(const double2* X, double2* Y, int64_t count, cudaStream_t st) {
  if (count) { k_copy<<<grid_for(count, 256), 256, 0, st>>>(X, Y, count); count_launch(); }
}

}  // namespace hz
