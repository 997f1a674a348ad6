// Flexible GMRES building blocks, one Krylov space per right-hand side
// (Sec. "Domain decomposition preconditioner": GMRES; K8 CGS2 Arnoldi, K10
// Givens least squares, K12 solution update).
//
// The basis vectors are complex blocks [n][s] in FP64 (outer solve) or FP32
// (the inner coarse solve of the mixed form). Dot products accumulate in the
// vector precision (or double-float) inside a lane and are summed over lanes,
// warps and CTAs in FP64 in a fixed order (deterministic); the Hessenberg
// matrix, the Givens rotations and the least-squares solve are FP64.
//
// One Arnoldi step: products V^H w with |w|^2, their sum over the CTAs (and
// which columns need a second pass), w -= V h, the second products, their sum,
// w -= V h, |w|^2, its sum with the Hessenberg column and the rotations, and
// v = w / |w|. GB300's FP64 pipe takes a warp's
// instruction every 64 clocks per scheduler, so that chains of FP64 sums by
// one thread are what dominates small blocks; they are spread over lanes and
// SMs, and so are the square roots and divisions of the per-column work.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "df.cuh"
#include "kernels.cuh"
#include "spmm.cuh"

namespace hz {

namespace {

__device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
template <typename V>
__device__ __forceinline__ V zero() {
  return mk((decltype(V::x))0, (decltype(V::x))0);
}
template <typename V>
__device__ __forceinline__ V from2(double2 a) {
  return mk((decltype(V::x))a.x, (decltype(V::x))a.y);
}
template <typename V>
__device__ __forceinline__ double2 to2(V a) {
  return make_double2((double)a.x, (double)a.y);
}
template <typename V>
__device__ __forceinline__ V cfms(V a, V b, V c) {  // c - a*b
  return mk(fma(-a.x, b.x, fma(a.y, b.y, c.x)), fma(-a.x, b.y, fma(-a.y, b.x, c.y)));
}
template <typename V>
__device__ __forceinline__ V cfma(V a, V b, V c) {  // c + a*b
  return mk(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
template <typename V>
__device__ __forceinline__ V conjmul_acc(V a, V b, V c) {  // c + conj(a)*b
  return mk(fma(a.x, b.x, fma(a.y, b.y, c.x)), fma(a.x, b.y, fma(-a.y, b.x, c.y)));
}
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 zsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 zdiv(double2 a, double2 b) {
  double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double zabs2(double2 a) { return a.x * a.x + a.y * a.y; }

inline unsigned grid_for(int64_t work, int block) { return (unsigned)((work + block - 1) / block); }

// Double-float operands (FP64 Krylov spaces of the mixed form with
// emulate_fp64): the basis stays in FP64 (the preconditioner reads it) and is
// split into FP32 pairs by its bit layout as it is read, so that it costs no
// second copy; w = A z is a double-float block.
__device__ __forceinline__ float4 df_split2(const double2 v) {
  const float2 r = df_split(v.x), i = df_split(v.y);
  return make_float4(r.x, r.y, i.x, i.y);
}
__device__ __forceinline__ float4 as_df(const float4 v) { return v; }
__device__ __forceinline__ float4 as_df(const double2 v) { return df_split2(v); }

// (reh, rel, imh, iml) += conj(v) w
__device__ __forceinline__ void df_conj_mac(float4& a, const float4 v, const float4 w) {
  df_mac(a.x, a.y, v.x, v.y, w.x, w.y);    // re += vr wr
  df_mac(a.x, a.y, v.z, v.w, w.z, w.w);    // re += vi wi
  df_mac(a.z, a.w, v.x, v.y, w.z, w.w);    // im += vr wi
  df_mac(a.z, a.w, -v.z, -v.w, w.x, w.y);  // im -= vi wr
}


}  // namespace

// ---------------------------------------------------------------------------
// Gram-Schmidt products: part[blk][i][c] = sum over the block's rows of
// conj(V_i[r][c]) W[r][c] for ni basis vectors and, as vector ni, |W_c|^2
// (norm = 1). Columns with mask[c] == 0 give zeros without reading their data.
//
// The two-level preconditioner carries a rounding difference of its inner
// Krylov iteration up by many orders of magnitude where the coarse mesh does
// not resolve the wavelength (1e-14 became 1e-4 of the result on the 5 Hz
// workload), so the order of every sum is part of the result: a CTA's row
// range is cut over NR / s threads per column, each adding its rows in turn,
// and the threads are added in turn in FP64. What is free is which threads do
// the work: up to DSLOT x DV vectors at a time, each slot of threads taking
// DV of them, so that W is read once for 12 vectors, all loads of a row are
// issued before its products, and the final sums of all vectors and columns
// run side by side (only the threads that had a row take part: one column of
// few rows used to add 256 parts one after the other, vector after vector).
// ---------------------------------------------------------------------------
constexpr int DV = 4;       // vectors per thread
constexpr int DSLOT = 3;    // vector slots per CTA: 12 vectors, 48 KB of parts
constexpr int NR = 256;     // threads per slot (whole columns of rows)
constexpr int DWARPS = 8;   // vectors per CTA of the sum over CTAs
constexpr size_t SMEM_MAX = 40960;  // shared memory of the per-column kernels at most

__device__ __forceinline__ void conj_mac(double2& a, double2 v, double2 w) { a = conjmul_acc(v, w, a); }
__device__ __forceinline__ void conj_mac(float2& a, float2 v, float2 w) { a = conjmul_acc(v, w, a); }
__device__ __forceinline__ void conj_mac(float4& a, float4 v, float4 w) { df_conj_mac(a, v, w); }
__device__ __forceinline__ double2 acc_d(double2 a) { return a; }
__device__ __forceinline__ double2 acc_d(float2 a) { return make_double2(a.x, a.y); }
__device__ __forceinline__ double2 acc_d(float4 a) {
  return make_double2(f2d(a.x) + f2d(a.y), f2d(a.z) + f2d(a.w));
}
template <bool DF, typename T>
__device__ __forceinline__ auto operand(T v) {
  if constexpr (DF)
    return as_df(v);
  else
    return v;
}
__device__ __forceinline__ void set_zero(double2& a) { a = make_double2(0.0, 0.0); }
__device__ __forceinline__ void set_zero(float2& a) { a = make_float2(0.f, 0.f); }
__device__ __forceinline__ void set_zero(float4& a) { a = make_float4(0.f, 0.f, 0.f, 0.f); }

template <bool DF, typename VB, typename VW>
__global__ void __launch_bounds__(NR* DSLOT) k_dots(const VB* __restrict__ Vb, int64_t vstride, int i0, int ni,
                                                    int norm, const VW* __restrict__ W, int64_t n, int s,
                                                    int64_t rows_per_blk, double2* __restrict__ part, int mstride,
                                                    const int* __restrict__ mask, int per) {
  using Op = decltype(operand<DF>(VW()));
  extern __shared__ double2 sh[];  // [vector][row thread][column]
  const int slot = threadIdx.y, nr = NR / s;
  const int rl = threadIdx.x / s, c = threadIdx.x - rl * s;
  const int nvec = min((int)blockDim.y * per, ni + norm - i0);
  const int v0 = i0 + slot * per, nq = min(per, nvec - slot * per);  // the slot's vectors
  const int qn = norm ? ni - v0 : DV;                                // the one that is W itself
  const int64_t r0 = blockIdx.x * rows_per_blk, rb = min(n, r0 + rows_per_blk);
  const int rows = (int)min((int64_t)nr, rb - r0);  // row threads with a row
  if (rl < rows) {
    Op acc[DV];
#pragma unroll
    for (int q = 0; q < DV; ++q) set_zero(acc[q]);
    const int64_t step = (int64_t)nr * s, e1 = (mask && !mask[c]) ? 0 : rb * s;
    const VB* pv = Vb + (int64_t)v0 * vstride;
#pragma unroll 2
    for (int64_t e = (r0 + rl) * s + c; e < e1; e += step) {
      const VW wr = W[e];
      VB v[DV];  // every load of the row before its products
#pragma unroll
      for (int q = 0; q < DV; ++q)
        if (q < nq && q != qn) v[q] = pv[q * vstride + e];
      const Op w = operand<DF>(wr);
#pragma unroll
      for (int q = 0; q < DV; ++q)
        if (q < nq) conj_mac(acc[q], q == qn ? w : operand<DF>(v[q]), w);
    }
#pragma unroll
    for (int q = 0; q < DV; ++q)
      if (q < nq) sh[(slot * per + q) * (nr * s) + threadIdx.x] = acc_d(acc[q]);
  }
  __syncthreads();
  for (int t = slot * blockDim.x + threadIdx.x; t < nvec * s; t += blockDim.x * blockDim.y) {
    const int v = t / s, x = t - v * s;
    double2 a = make_double2(0.0, 0.0);
    for (int l = 0; l < rows; ++l) a = zadd(a, sh[v * (nr * s) + l * s + x]);
    part[((int64_t)blockIdx.x * mstride + i0 + v) * s + x] = a;
  }
}

// Per-column data of a Krylov space, as the kernels read it
struct ColState {
  int s, m, j;
  double2 *h1, *h2;     // [m+1][s]
  float4* hdf;          // coefficients in double-float, or NULL
  double2* nrm;         // [s] |w|^2 before the step (first pass)
  int* reorth;          // [s]
  double2 *H, *Hraw;    // [s][(m+1) m]
  double* cs;
  double2 *sn, *g;
  double *beta, *res, *out;
  const double* tol;
  int *kc, *done;
  int* count;           // [s] finished CTAs per column, back to zero after every launch
  int inplace;          // RED_FINISH works in the arrays themselves
};

// Column j of the Hessenberg matrix, the previous Givens rotations, the new
// one, the rotated right-hand side g and the residual estimate |g_{j+1}|: one
// warp per column, `nrm2` = |w|^2 after the updates.
__device__ void arnoldi_column(const ColState& K, int c, double nrm2, double2* Hs, double* cs, double2* sn) {
  const int lane = threadIdx.x, s = K.s, m = K.m, j = K.j;
  const double hb = sqrt(nrm2);
  double hn2 = 0.0;
  for (int i = lane; i <= j; i += 32) {
    const double2 h = zadd(K.h1[i * s + c], K.h2[i * s + c]);
    Hs[i] = h;
    hn2 += zabs2(h);
    if (i < j) {
      cs[i] = K.cs[c * m + i];
      sn[i] = K.sn[c * m + i];
    }
  }
  for (int o = 16; o > 0; o >>= 1) hn2 += __shfl_xor_sync(0xffffffffu, hn2, o);
  hn2 += hb * hb;
  const bool breakdown = !(hb > 1e-14 * sqrt(hn2));
  const bool done = K.done[c] != 0;
  __syncwarp();
  if (lane == 0) {
    K.beta[c] = breakdown ? 0.0 : 1.0 / hb;
    Hs[j + 1] = make_double2(breakdown ? 0.0 : hb, 0.0);
  }
  if (done) return;
  double2* Hc = K.H + (int64_t)c * (m + 1) * m + (int64_t)j * (m + 1);
  __syncwarp();
  if (K.Hraw) {  // the unrotated column (recycling reads it after the cycle)
    double2* Hr = K.Hraw + (int64_t)c * (m + 1) * m + (int64_t)j * (m + 1);
    for (int i = lane; i <= j + 1; i += 32) Hr[i] = Hs[i];
    __syncwarp();
  }
  if (lane == 0) {
    double2 a = Hs[0];
    for (int i = 0; i < j; ++i) {
      const double2 b = Hs[i + 1];
      Hs[i] = zadd(make_double2(cs[i] * a.x, cs[i] * a.y), zmul(sn[i], b));
      a = zsub(make_double2(cs[i] * b.x, cs[i] * b.y), zmul(make_double2(sn[i].x, -sn[i].y), a));
    }
    const double2 b = Hs[j + 1];
    const double aa = sqrt(zabs2(a)), bb = sqrt(zabs2(b));
    double cj;
    double2 sj;
    if (bb == 0.0) {
      cj = 1.0;
      sj = make_double2(0.0, 0.0);
    } else if (aa == 0.0) {
      cj = 0.0;
      sj = make_double2(b.x / bb, -b.y / bb);
    } else {
      const double tt = sqrt(aa * aa + bb * bb);
      cj = aa / tt;
      sj = zmul(make_double2(a.x / aa, a.y / aa), make_double2(b.x / tt, -b.y / tt));
    }
    K.cs[c * m + j] = cj;
    K.sn[c * m + j] = sj;
    Hs[j] = zadd(make_double2(cj * a.x, cj * a.y), zmul(sj, b));
    Hs[j + 1] = make_double2(0.0, 0.0);
    double2* gc = K.g + c * (m + 1);
    const double2 gj = gc[j];
    gc[j] = make_double2(cj * gj.x, cj * gj.y);
    const double2 gn = zmul(make_double2(-sj.x, sj.y), gj);
    gc[j + 1] = gn;
    K.kc[c] = j + 1;
    const double r = sqrt(zabs2(gn));
    K.res[c] = r;
    if (r <= K.tol[c] || breakdown) K.done[c] = 1;
  }
  __syncwarp();
  for (int i = lane; i <= j + 1; i += 32) Hc[i] = Hs[i];
}

// What a sum over the CTAs is followed by
enum { RED_H1, RED_H2, RED_FINISH, RED_START, RED_NORM };

// Sums over the nblk CTAs of part[blk][v][c], v < nvec: CTA (column, 8
// vectors), a warp per vector.
//   RED_H1     h1 and |w|^2 (vector nvec - 1); the last CTA of a column decides
//              on its second Gram-Schmidt pass, needed only where the first one
//              cancelled: with w the vector before and w' after it, |w'|^2 =
//              |w|^2 - sum |h_i|^2; again when |w'|^2 < |w|^2 / 2 ("twice is enough")
//   RED_H2     h2
//   RED_FINISH |w|^2, then the column's Hessenberg and rotation work
//   RED_START  beta = |r|, g = beta e_1, flags
//   RED_NORM   out = |x|
template <int MODE>
__global__ void k_reduce(const double2* __restrict__ part, int nblk, int nvec, int mstride, ColState K) {
  extern __shared__ double2 dyn[];
  const int lane = threadIdx.x & 31, v = blockIdx.y * DWARPS + (threadIdx.x >> 5), c = blockIdx.x, s = K.s;
  double2 a = make_double2(0.0, 0.0);
  if (v < nvec) {
    for (int b = lane; b < nblk; b += 32) a = zadd(a, part[((int64_t)b * mstride + v) * s + c]);
    for (int o = 16; o > 0; o >>= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
      a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
    }
  }
  if (MODE == RED_NORM) {
    if (lane == 0) K.out[c] = sqrt(a.x);
  } else if (MODE == RED_START) {
    const double b = sqrt(a.x);
    for (int i = lane; i <= K.m; i += 32) K.g[c * (K.m + 1) + i] = make_double2(i == 0 ? b : 0.0, 0.0);
    if (lane == 0) {
      K.kc[c] = 0;
      K.res[c] = b;
      K.done[c] = (b <= K.tol[c]) ? 1 : 0;
      K.beta[c] = b > 0.0 ? 1.0 / b : 0.0;
    }
  } else if (MODE == RED_FINISH) {
    // scratch in shared memory, or for a restart length that does not fit the arrays in place (a
    // finished column's entries are not used again)
    double2* Hs = K.inplace ? K.H + (int64_t)c * (K.m + 1) * K.m + (int64_t)K.j * (K.m + 1) : dyn;
    double2* sn = K.inplace ? K.sn + (int64_t)c * K.m : dyn + K.m + 1;
    double* cs = K.inplace ? K.cs + (int64_t)c * K.m : reinterpret_cast<double*>(dyn + 2 * K.m + 1);
    arnoldi_column(K, c, a.x, Hs, cs, sn);
  } else {
    const int ni = MODE == RED_H1 ? nvec - 1 : nvec;
    if (lane == 0 && v < ni) {
      (MODE == RED_H1 ? K.h1 : K.h2)[v * s + c] = a;
      if (K.hdf) K.hdf[v * s + c] = df_split2(a);
    }
    if (MODE == RED_H1) {
      if (lane == 0 && v == ni) K.nrm[c] = a;
      __shared__ int last;
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) last = atomicInc((unsigned*)K.count + c, gridDim.y - 1) == gridDim.y - 1;
      __syncthreads();
      if (last && threadIdx.x < 32) {
        __threadfence();
        double hh = 0.0;
        for (int i = lane; i < ni; i += 32) hh += zabs2(__ldcg(K.h1 + i * s + c));
        for (int o = 16; o > 0; o >>= 1) hh += __shfl_xor_sync(0xffffffffu, hh, o);
        const double ww = __ldcg(&K.nrm[c].x);
        if (lane == 0) K.reorth[c] = (ww - hh < 0.5 * ww) ? 1 : 0;
      }
    }
  }
}

// W[r][c] -= sum_{i<ni} V_i[r][c] h[i][c] (columns with mask[c] == 0 stay);
// threads are (column, row) pairs
__device__ __forceinline__ void cfms_w(double2& w, double2 v, double2 h) { w = cfms(v, h, w); }
__device__ __forceinline__ void cfms_w(float2& w, float2 v, double2 h) { w = cfms(v, from2<float2>(h), w); }
__device__ __forceinline__ void cfms_w(float4& w, float4 v, float4 h) {
  df_mac(w.x, w.y, -v.x, -v.y, h.x, h.y);  // re -= vr hr
  df_mac(w.x, w.y, v.z, v.w, h.z, h.w);    // re += vi hi
  df_mac(w.z, w.w, -v.x, -v.y, h.z, h.w);  // im -= vr hi
  df_mac(w.z, w.w, -v.z, -v.w, h.x, h.y);  // im -= vi hr
}
__device__ __forceinline__ void settle(double2&) {}
__device__ __forceinline__ void settle(float2&) {}
__device__ __forceinline__ void settle(float4& w) {
  df_norm(w.x, w.y);
  df_norm(w.z, w.w);
}
template <bool DF, typename VB, typename VW, typename VH>
__global__ void __launch_bounds__(256) k_update(const VB* __restrict__ Vb, int64_t vstride, int ni,
                                                const VH* __restrict__ h, VW* __restrict__ W, int64_t n, int s,
                                                const int* __restrict__ mask) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.y + threadIdx.y;
  const int c = threadIdx.x;
  if (r >= n || (mask && !mask[c])) return;
  const int64_t g = r * s + c;
  VW w = W[g];
#pragma unroll 4
  for (int i = 0; i < ni; ++i) cfms_w(w, operand<DF>(Vb[i * vstride + g]), h[i * s + c]);
  settle(w);
  W[g] = w;
}

template <typename V>
__global__ void k_scale_cols(const V* __restrict__ X, const double* __restrict__ sc, V* __restrict__ Y, int64_t n,
                             int s) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.y + threadIdx.y;
  if (r >= n) return;
  const int64_t g = r * s + threadIdx.x;
  const auto a = (decltype(V::x))sc[threadIdx.x];
  const V x = X[g];
  Y[g] = mk(a * x.x, a * x.y);
}
// v = w beta[c] (double-float product, stored in FP64)
__global__ void k_scale_cols(const float4* __restrict__ X, const double* __restrict__ beta, double2* __restrict__ Y,
                             int64_t n, int s) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.y + threadIdx.y;
  if (r >= n) return;
  const int64_t g = r * s + threadIdx.x;
  const float2 b = df_split(beta[threadIdx.x]);
  const float4 x = X[g];
  float4 y;
  df_mul(y.x, y.y, x.x, x.y, b.x, b.y);
  df_mul(y.z, y.w, x.z, x.w, b.x, b.y);
  Y[g] = make_double2(df_join(y.x, y.y), df_join(y.z, y.w));
}

// y = R^{-1} g per column (R = rotated Hessenberg, kc[c] steps): one warp per
// column brings R and g to shared memory, one lane substitutes back (R stays
// in place when it does not fit)
__global__ void k_ls_solve(int m, const double2* __restrict__ H, const double2* __restrict__ g,
                           const int* __restrict__ kc, double2* __restrict__ y, int inplace) {
  extern __shared__ double2 dyn[];  // [m][m] R by columns, then y
  const int c = blockIdx.x, lane = threadIdx.x, k = kc[c];
  const double2* Hc = H + (int64_t)c * (m + 1) * m;
  const double2* gc = g + (int64_t)c * (m + 1);
  double2* yc = y + (int64_t)c * m;
  const int ld = inplace ? m + 1 : m;
  const double2* R = inplace ? Hc : dyn;
  if (!inplace) {
    for (int e = lane; e < k * k; e += 32) {
      const int l = e / k, i = e - l * k;
      dyn[i + l * m] = Hc[i + (int64_t)l * (m + 1)];
    }
    __syncwarp();
  }
  double2* ys = inplace ? yc : dyn + m * m;
  if (lane == 0)
    for (int i = k - 1; i >= 0; --i) {
      double2 v = gc[i];
      for (int l = i + 1; l < k; ++l) v = zsub(v, zmul(R[i + (int64_t)l * ld], ys[l]));
      const double2 d = R[i + (int64_t)i * ld];
      ys[i] = (d.x == 0.0 && d.y == 0.0) ? make_double2(0.0, 0.0) : zdiv(v, d);
    }
  if (!inplace) {
    __syncwarp();
    for (int i = lane; i < k; i += 32) yc[i] = ys[i];
  }
}

template <typename V>
__global__ void k_sol_update(const V* __restrict__ Zk, int64_t vstride, const double2* __restrict__ y,
                             const int* __restrict__ kc, V* __restrict__ X, int64_t n, int s, int m) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.y + threadIdx.y;
  if (r >= n) return;
  const int c = threadIdx.x;
  const int64_t g = r * s + c;
  V x = X[g];
  const int k = kc[c];
  for (int j = 0; j < k; ++j) x = cfma(Zk[j * vstride + g], from2<V>(y[c * m + j]), x);
  X[g] = x;
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static ColState col_state(const DevKrylov& K, int j) {
  ColState S;
  S.s = K.s;
  S.m = K.m;
  S.j = j;
  S.h1 = K.h1;
  S.h2 = K.h2;
  S.hdf = K.df ? K.hdf : nullptr;
  S.nrm = K.h2 + (int64_t)K.m * K.s;  // row m of h2: a step uses rows 0..m-1
  S.reorth = K.reorth;
  S.H = K.H;
  S.Hraw = K.Hraw;
  S.cs = K.cs;
  S.sn = K.sn;
  S.g = K.g;
  S.beta = K.beta;
  S.res = K.res;
  S.out = nullptr;
  S.tol = K.tol;
  S.kc = K.kc;
  S.done = K.done;
  S.count = K.count;
  S.inplace = (size_t)(2 * K.m + 1) * sizeof(double2) + (size_t)K.m * sizeof(double) > SMEM_MAX;
  return S;
}

// threads of an element-wise kernel: (column, row)
static dim3 row_block(int s) { return dim3(s, std::max(1, 256 / s)); }

// Products of W with ni basis vectors (and with itself); returns the CTAs
// whose parts have to be added.
template <bool DF, typename VB, typename VW>
static int dots(DevKrylov& K, const VB* Vb, int64_t vstride, int ni, int norm, const VW* W, const int* mask,
                cudaStream_t st) {
  const int s = K.s, nvec = ni + norm, threads = (NR / s) * s;
  const int64_t rpb = (K.n + K.nblk - 1) / K.nblk;
  const int nb = (int)((K.n + rpb - 1) / rpb);
  for (int i0 = 0; i0 < nvec; i0 += DSLOT * DV) {
    const int nv = std::min(DSLOT * DV, nvec - i0), slots = (nv + DV - 1) / DV, per = (nv + slots - 1) / slots;
    k_dots<DF, VB, VW><<<nb, dim3(threads, slots), (size_t)slots * per * threads * sizeof(double2), st>>>(
        Vb, vstride, i0, ni, norm, W, K.n, s, rpb, K.hpart, K.m + 2, mask, per);
    count_launch();
  }
  return nb;
}

template <int MODE>
static void reduce(const DevKrylov& K, const ColState& S, int nblk, int nvec, cudaStream_t st) {
  const bool one = MODE >= RED_FINISH;
  size_t shm = MODE == RED_FINISH ? (size_t)(2 * K.m + 1) * sizeof(double2) + (size_t)K.m * sizeof(double) : 0;
  if (shm > SMEM_MAX) shm = 0;
  k_reduce<MODE><<<dim3(K.s, one ? 1 : (nvec + DWARPS - 1) / DWARPS), one ? 32 : 32 * DWARPS, shm, st>>>(
      K.hpart, nblk, nvec, K.m + 2, S);
  count_launch();
}

template <bool DF, typename V>
static void column_norms_t(const V* X, double* out, DevKrylov& K, cudaStream_t st) {
  const int nb = dots<DF>(K, X, 0, 0, 1, X, nullptr, st);
  ColState S = col_state(K, 0);
  S.out = out;
  reduce<RED_NORM>(K, S, nb, 1, st);
}

template <bool DF, typename V>
static void krylov_start_t(DevKrylov& K, const V* R, cudaStream_t st) {
  const int nb = dots<DF>(K, R, 0, 0, 1, R, nullptr, st);
  reduce<RED_START>(K, col_state(K, 0), nb, 1, st);
  const dim3 b = row_block(K.s);
  { k_scale_cols<V><<<grid_for(K.n, b.y), b, 0, st>>>(R, K.beta, (V*)K.V, K.n, K.s); count_launch(); }
}

template <bool DF, typename V, typename VW, typename VH>
static void krylov_arnoldi_t(DevKrylov& K, int j, VW* W, const VH* ha, const VH* hb, cudaStream_t st) {
  const int64_t vs = K.n * K.s;
  V* Vb = (V*)K.V;
  const ColState S = col_state(K, j);
  const dim3 b = row_block(K.s);
  int nb = dots<DF>(K, Vb, vs, j + 1, 1, W, nullptr, st);
  reduce<RED_H1>(K, S, nb, j + 2, st);
  { k_update<DF, V, VW, VH><<<grid_for(K.n, b.y), b, 0, st>>>(Vb, vs, j + 1, ha, W, K.n, K.s, nullptr); count_launch(); }
  nb = dots<DF>(K, Vb, vs, j + 1, 0, W, K.reorth, st);
  reduce<RED_H2>(K, S, nb, j + 1, st);
  { k_update<DF, V, VW, VH><<<grid_for(K.n, b.y), b, 0, st>>>(Vb, vs, j + 1, hb, W, K.n, K.s, K.reorth); count_launch(); }
  nb = dots<DF>(K, (const V*)nullptr, 0, 0, 1, W, nullptr, st);
  reduce<RED_FINISH>(K, S, nb, 1, st);
  { k_scale_cols<<<grid_for(K.n, b.y), b, 0, st>>>((const VW*)W, K.beta, Vb + (int64_t)(j + 1) * vs, K.n, K.s);
    count_launch(); }
}

template <typename V>
static void krylov_update_t(DevKrylov& K, V* X, cudaStream_t st) {
  const dim3 b = row_block(K.s);
  const size_t shm = (size_t)K.m * (K.m + 1) * sizeof(double2);
  const bool fits = shm <= SMEM_MAX;
  { k_ls_solve<<<K.s, 32, fits ? shm : 0, st>>>(K.m, K.H, K.g, K.kc, K.y, !fits); count_launch(); }
  { k_sol_update<V><<<grid_for(K.n, b.y), b, 0, st>>>((const V*)K.Zk, K.n * K.s, K.y, K.kc, X, K.n, K.s, K.m); count_launch(); }
}

void column_norms(const void* X, int64_t, int, double* out, DevKrylov& K, cudaStream_t st) {
  if (K.fp32)
    column_norms_t<false>((const float2*)X, out, K, st);
  else if (K.df)
    column_norms_t<true>((const double2*)X, out, K, st);
  else
    column_norms_t<false>((const double2*)X, out, K, st);
}
void krylov_start(DevKrylov& K, const void* R, cudaStream_t st) {
  if (K.fp32)
    krylov_start_t<false>(K, (const float2*)R, st);
  else if (K.df)
    krylov_start_t<true>(K, (const double2*)R, st);
  else
    krylov_start_t<false>(K, (const double2*)R, st);
}
void krylov_arnoldi(DevKrylov& K, int j, cudaStream_t st) {
  if (K.df)
    krylov_arnoldi_t<true, double2>(K, j, K.Wdf, (const float4*)K.hdf, (const float4*)K.hdf, st);
  else if (K.fp32)
    krylov_arnoldi_t<false, float2>(K, j, (float2*)K.W, (const double2*)K.h1, (const double2*)K.h2, st);
  else
    krylov_arnoldi_t<false, double2>(K, j, (double2*)K.W, (const double2*)K.h1, (const double2*)K.h2, st);
}
void krylov_update(DevKrylov& K, void* X, cudaStream_t st) {
  if (K.fp32) {
    krylov_update_t<float2>(K, (float2*)X, st);
  } else {
    krylov_update_t<double2>(K, (double2*)X, st);
  }
}

// ---------------------------------------------------------------------------
// FP32 coarse-level helpers (mixed form): SpMM with float values, precision casts
// ---------------------------------------------------------------------------
namespace {
struct OutRowsF {  // Y = A X, or B - A X
  float2* Y;
  const float2* B;
  int s;
  __device__ __forceinline__ void operator()(int64_t r, int c, float2 y) const {
    const int64_t g = r * s + c;
    if (B) {
      const float2 b = B[g];
      y = make_float2(b.x - y.x, b.y - y.y);
    }
    Y[g] = y;
  }
};
}  // namespace

void spmm_split_f32(const DevSplitCsr& A, const float2* X, float2* Y, int s, cudaStream_t st, const float2* B) {
  spmm_launch<SpF32, true>(A.n, s, A.rp_re, A.col_re, A.val_re_f, A.rp_im, A.col_im, A.val_im_f, X, OutRowsF{Y, B, s}, st);
}
void spmm_real_f32(int64_t nrows, const int64_t* rp, const int32_t* col, const float* val, const float2* X,
                   float2* Y, int s, cudaStream_t st) {
  spmm_launch<SpF32, true>(nrows, s, rp, col, val, nullptr, nullptr, nullptr, X, OutRowsF{Y, nullptr, s}, st);
}

__global__ void k_d2f(const double2* __restrict__ X, float2* __restrict__ Y, int64_t count) {
  int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g < count) Y[g] = make_float2((float)X[g].x, (float)X[g].y);
}
__global__ void k_f2d(const float2* __restrict__ X, double2* __restrict__ Y, int64_t count) {
  int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g < count) Y[g] = make_double2(X[g].x, X[g].y);
}
void cast_d2f(const double2* X, float2* Y, int64_t count, cudaStream_t st) {
  if (count) { k_d2f<<<grid_for(count, 256), 256, 0, st>>>(X, Y, count); count_launch(); }
}
void cast_f2d(const float2* X, double2* Y, int64_t count, cudaStream_t st) {
  if (count) { k_f2d<<<grid_for(count, 256), 256, 0, st>>>(X, Y, count); count_launch(); }
}

}  // namespace hz
