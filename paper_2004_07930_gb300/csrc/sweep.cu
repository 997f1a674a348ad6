// Front sweeps: the solves with the factored local matrices A_i (the paper's
// direct local solver inside Eq. oras), on the partitioned inverse that
// factor.cu stores.
//
// Per front t of order f with k pivots, X_t = [L11^{-1}; -L21 L11^{-1}]
// (f x k) and 1/D turn the solve into two products without a recurrence
// inside the front:
//   forward  (leaves to root): t = X_t b_P;  y_P = t[0:k] / D;
//                              parent update  w = c_U + t[k:f]
//   backward (root to leaves): x_P = X_t^T [y_P; x_U]
// where b_P is the sub-vector at the pivots plus the children's updates that
// land there, c_U the children's updates on the other rows.
//
// Work split. The output rows of a front are cut into groups of MF_GR = 16.
// One warp computes one group for up to 16 right-hand sides: a lane keeps
// RPT rows x CPT columns of complex accumulators (4 x 2 at 16 columns: 16
// packed FMA for two loads of factor entries and one of input values), and
// all the lanes of a row read or write 128 contiguous bytes of it. A CTA of four
// warps takes a task: a run of groups of one front, whose input rows are
// staged once in shared memory, MF_CHUNK reduction indices at a time. Wider
// blocks run as several column blocks of 16, side by side in the grid so
// that the factor entries are read from L2 after the first.
//
// Factor layout (factor.cu writes it): group after group, each as
// [reduction index][row of the group], the row count padded to 4, without
// the structural zeros: group g of X_t keeps its columns below
// min(k, 16 (g + 1)), group g of X_t^T its columns from 16 g on. A warp
// therefore streams one contiguous range, through its own ring of
// cp.async stages, one stage ahead of the products, starting before the
// previous launch of the sweep has finished.
//
// What bounds it: on the 5 Hz workload (0.95M dofs, 64 subdomains, 16
// columns) the FP32 FMA pipe: 444M factor entries, 114 GFLOP per
// application, 1.5 ms at the pipe's 74.8 TFLOP/s; with one column HBM: 7.1 GB,
// 1.05 ms. Measured, whole preconditioner: 4.05 ms (tiles of 128 rows,
// one or a quarter of one per thread: 7.16) and 1.66 ms (2.00). With one column
// eight of a warp's lanes hold distinct rows and each row's sum is one chain
// in order, so that short levels wait for that chain (see k_sweep_long). The leaf level runs at
// 52-55 % of the pipe; the middle levels, 1-10 K small fronts each, spend
// 30-55 us on the latency of task, indices, inputs and factors in turn.
//
// FP64 has one pipe per scheduler that takes a warp's multiply-add every 64
// clocks (1.2 TFLOP/s over the 608 schedulers), so that a short level must
// reach all of them: its tasks are single groups, and the four warps share
// the group's reduction stage by stage (KS), summing their parts at the end.
//
// Order of the sums. The reduction of every output entry is sequential
// inside a chunk and the chunks are added in order (FP64 single groups: four
// parts in order); neither depends on the launch form or the block width.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "kernels.cuh"

#include "cplx.cuh"
#include "f32x2.cuh"

namespace hz {

namespace {

constexpr int SW_THREADS = 32 * SW_NW;
constexpr int SW_NST = 2;  // ring stages per warp

// Ring stages: 2-3 KB where the whole input is staged first (levels of many
// small fronts: more CTAs per SM; the forward sweep's inputs are the smaller
// ones), 4 KB where the input streams by (long reductions: fewer stage turns)
template <typename V, bool FWD, bool STREAM>
struct SwV {
  static constexpr int BYTES = STREAM ? 4096 : (FWD ? 3072 : 2048);
  static constexpr int KC = BYTES / (MF_GR * (int)sizeof(V));  // reduction indices per stage
  static constexpr int STAGE = KC * MF_GR;                     // entries per stage
};

// Lanes of a warp: CL lanes share a row, each with CPT columns; RG row sets of
// up to RPT rows each. FP32 works on row pairs (packed multiply-adds). FP64
// with one column gives the real and the imaginary part to two lanes.
// Staging: a thread moves SPT columns (FP32: 16 bytes) of a row, RPP rows per
// pass of the CTA, U passes (CH rows) at a time where the input streams by.
template <typename V, int S, bool FWD>
struct SwS {
  static constexpr bool F32 = sizeof(V) == 8;
  static constexpr bool SPLIT = !F32 && S == 1;
  static constexpr int RPT = F32 ? (S == 16 ? 4 : 2) : (S == 16 ? 4 : (S == 8 ? 2 : 1));
  static constexpr int CPT = F32 ? (S >= 8 ? 2 : 1) : (S >= 4 ? 2 : 1);
  static constexpr int CL = SPLIT ? 2 : S / CPT;
  static constexpr int RG = MF_GR / RPT;  // FP64: row sets of a warp
  static constexpr int SPT = F32 ? (S >= 2 ? 2 : 1) : CPT;
  static constexpr int CLS = S / SPT;
  static constexpr int RPP = SW_THREADS / CLS;
  static constexpr int WANT = F32 && !FWD ? 64 : 32;  // the forward rows pass through registers
  static constexpr int U = RPP < WANT ? WANT / RPP : 1;
  static constexpr int CH = U * RPP;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
// -x by its sign bit: a negation that a select keeps apart from the
// multiply-add is an instruction of the FP64 pipe, every third one of the
// one-column loop (quarter workload, FP64, one column: 3.47 -> 2.14 ms; the
// tiles before these sweeps 2.87).
__device__ __forceinline__ double neg_bits(double x) {
  return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}
// t / D. The two forms round the imaginary part differently in the last bit;
// rows whose reduction spans several chunks have always used the second, and
// keep it so that results stay the same to the bit.
template <bool SPLIT, typename V>
__device__ __forceinline__ V mul_dinv(V a, V b) {
  return mk2(fma_rn(a.x, b.x, -mul_rn(a.y, b.y)),
             SPLIT ? fma_rn(a.y, b.x, mul_rn(a.x, b.y)) : fma_rn(a.x, b.y, mul_rn(a.y, b.x)));
}

// CPT values of one row (rows are padded to the sweep's column blocks, see
// sweep_cols: aligned and always whole), read through L2: other CTAs write them
template <int CPT>
__device__ __forceinline__ void ld_cols(const float2* p, float2 (&v)[CPT]) {
  if constexpr (CPT == 2) {
    const float4 q = __ldcg(reinterpret_cast<const float4*>(p));
    v[0] = make_float2(q.x, q.y);
    v[1] = make_float2(q.z, q.w);
  } else {
    v[0] = __ldcg(p);
  }
}
template <int CPT>
__device__ __forceinline__ void ld_cols(const double2* p, double2 (&v)[CPT]) {
#pragma unroll
  for (int q = 0; q < CPT; ++q) v[q] = __ldcg(p + q);
}
template <int CPT>
__device__ __forceinline__ void st_cols(float2* p, const float2 (&v)[CPT]) {
  if constexpr (CPT == 2)
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  else
    p[0] = v[0];
}
template <int CPT>
__device__ __forceinline__ void st_cols(double2* p, const double2 (&v)[CPT]) {
#pragma unroll
  for (int q = 0; q < CPT; ++q) p[q] = v[q];
}

template <typename V>
struct SweepArgs {
  const SweepTask* tasks;
  const int* rows;     // sub-vector row of each front row
  const int2* csrc;    // the (up to two) child update rows landing on each front row
  const V* M;          // grouped X_t (forward) or X_t^T (backward)
  const V* Dinv;
  V* Xsub;
  V* Wout;
  int s;               // row length of Xsub and Wout (sweep_cols)
  int kids;            // some front of the level has children
};

// A lane's accumulators, RPT rows x CPT columns
template <typename V, int S>
struct SwAcc;
template <int S>
struct SwAcc<float2, S> {
  using L = SwS<float2, S, true>;
  static constexpr int P = L::RPT / 2, CPT = L::CPT;
  pair2 re[P][CPT], im[P][CPT];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int q = 0; q < CPT; ++q) re[p][q] = im[p][q] = 0;
  }
  __device__ __forceinline__ void add(const SwAcc& o) {
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int q = 0; q < CPT; ++q) {
        re[p][q] = add2(re[p][q], o.re[p][q]);
        im[p][q] = add2(im[p][q], o.im[p][q]);
      }
  }
  // row i, column q (constant after unrolling)
  __device__ __forceinline__ float2 get(int i, int q) const {
    const float2 r = unpk(re[i / 2][q]), m = unpk(im[i / 2][q]);
    return i % 2 ? make_float2(r.y, m.y) : make_float2(r.x, m.x);
  }
  // rows per lane of a group of nrp padded rows
  static __device__ __forceinline__ int rows(int nrp) { return S == 16 && nrp <= 8 ? 2 : L::RPT; }

  template <int NP, int NRP>
  __device__ __forceinline__ void mac_n(const float2* a, const float2* b, int n, int rg) {
    if (rg * 2 * NP < NRP) a += rg * 2 * NP;
    auto step = [&](const float2* ak, const float2* bk) {
      float2 bv[CPT];
      if constexpr (CPT == 2) {
        const float4 t = *reinterpret_cast<const float4*>(bk);
        bv[0] = make_float2(t.x, t.y);
        bv[1] = make_float2(t.z, t.w);
      } else {
        bv[0] = *bk;
      }
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const float4 t = *reinterpret_cast<const float4*>(ak + 2 * p);
        const pair2 ar = pk(t.x, t.y), ai = pk(t.z, t.w);
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
          const pair2 br = pk(bv[q].x, bv[q].x), bi = pk(bv[q].y, bv[q].y), nbi = pk(-bv[q].y, -bv[q].y);
          re[p][q] = fma2(ar, br, fma2(ai, nbi, re[p][q]));
          im[p][q] = fma2(ar, bi, fma2(ai, br, im[p][q]));
        }
      }
    };
    int kk = 0;
#pragma unroll 1
    for (; kk + 4 <= n; kk += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) step(a + u * NRP, b + u * S);
      a += 4 * NRP;
      b += 4 * S;
    }
#pragma unroll 1
    for (; kk < n; ++kk) {
      step(a, b);
      a += NRP;
      b += S;
    }
  }
  // += (factor stage) x (staged inputs): n reduction indices of a group of nrp padded rows
  __device__ __forceinline__ void mac(const float2* a, const float2* b, int n, int nrp, int rg, int) {
    if (nrp == 16)
      mac_n<P, 16>(a, b, n, rg);
    else if (nrp == 12)
      mac_n<P, 12>(a, b, n, rg);
    else if (nrp == 8)
      mac_n<1, 8>(a, b, n, rg);
    else
      mac_n<1, 4>(a, b, n, rg);
  }
};
template <int S>
struct SwAcc<double2, S> {
  using L = SwS<double2, S, true>;
  static constexpr int RPT = L::RPT, CPT = L::CPT, RG = L::RG;
  double2 v[RPT][CPT];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
      for (int q = 0; q < CPT; ++q) v[i][q] = make_double2(0.0, 0.0);
  }
  __device__ __forceinline__ void add(const SwAcc& o) {
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
      for (int q = 0; q < CPT; ++q) v[i][q] = c_add(v[i][q], o.v[i][q]);
  }
  __device__ __forceinline__ double2 get(int i, int q) const {
    if constexpr (L::SPLIT) {  // the even lane's real part and the odd lane's imaginary part
      const double m = v[i][q].x, o = __shfl_xor_sync(0xffffffffu, m, 1);
      return threadIdx.x & 1 ? make_double2(o, m) : make_double2(m, o);
    } else {
      return v[i][q];
    }
  }
  static __device__ __forceinline__ int rows(int nrp) { return (nrp + RG - 1) / RG; }

  template <int N>
  __device__ __forceinline__ void mac_n(const double2* a, const double2* b, int n, int nrp, int rg, int lane) {
    if (rg * N < nrp) a += rg * N;
    if constexpr (L::SPLIT) {
#pragma unroll 4
      for (int kk = 0; kk < n; ++kk, a += nrp, ++b) {
        const double2 av = *a, bv = *b;
        const double b1 = lane & 1 ? bv.y : bv.x, b2 = lane & 1 ? bv.x : neg_bits(bv.y);
        v[0][0].x = fma(av.x, b1, fma(av.y, b2, v[0][0].x));
      }
    } else {
#pragma unroll 4
      for (int kk = 0; kk < n; ++kk, a += nrp, b += S) {
        double2 bv[CPT];
#pragma unroll
        for (int q = 0; q < CPT; ++q) bv[q] = b[q];
#pragma unroll
        for (int i = 0; i < N; ++i) {
          const double2 av = a[i];
#pragma unroll
          for (int q = 0; q < CPT; ++q) v[i][q] = c_fma(av, bv[q], v[i][q]);
        }
      }
    }
  }
  __device__ __forceinline__ void mac(const double2* a, const double2* b, int n, int nrp, int rg, int lane) {
    const int r = rows(nrp);
    if (RPT == 1 || r == 1)
      mac_n<1>(a, b, n, nrp, rg, lane);
    else if (RPT == 2 || r == 2)
      mac_n<(RPT < 2 ? 1 : 2)>(a, b, n, nrp, rg, lane);
    else if (r == 3)
      mac_n<(RPT < 3 ? 1 : 3)>(a, b, n, nrp, rg, lane);
    else
      mac_n<RPT>(a, b, n, nrp, rg, lane);
  }
};

// One task for columns [c0, c0 + S) of the block. Its input rows are staged
// whole, or (STREAM) CH rows at a time in two buffers, the next rows loaded
// while the current ones are used.
// `wait` is called once, after the loads that only need set-up data have been
// issued and before the first load of data that earlier levels write; it
// returns false (to every thread) when the wait was given up, and then the
// task is abandoned.
// KS: the warps share the task's single group, warp w taking its stages w,
// w + SW_NW, ...
template <typename V, int S, bool FWD, bool STREAM, bool KS, typename Wait>
__device__ __forceinline__ bool sweep_task_t(const SweepArgs<V>& A, const SweepTask& T, int c0, unsigned char* smem,
                                           Wait&& wait) {
  using L = SwS<V, S, FWD>;
  constexpr int CPT = L::CPT, SPT = L::SPT, CL = L::CL, CLS = L::CLS, RPT = L::RPT;
  constexpr int KC = KS ? 2048 / (MF_GR * (int)sizeof(V)) : SwV<V, FWD, STREAM>::KC;  // KS: the same in every form
  constexpr int STAGE = SwV<V, FWD, STREAM>::STAGE, BYTES = SwV<V, FWD, STREAM>::BYTES;
  constexpr int U = L::U, RPP = L::RPP, CH = L::CH;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int s = A.s;
  V* ring = reinterpret_cast<V*>(smem) + (size_t)warp * SW_NST * STAGE;
  V* bs = reinterpret_cast<V*>(smem + (size_t)SW_NW * SW_NST * BYTES);  // [rows][S]
  const int k = T.k, f = T.f, nout = FWD ? f : k;
  const int gend = T.g0 + T.ng;
  // reduction range of the task's groups
  const int lo = FWD ? 0 : MF_GR * T.g0;
  const int hi = FWD ? min(k, MF_GR * gend) : f;
  const int rg = lane / CL, col = L::SPLIT ? 0 : (lane % CL) * CPT;  // lane's row set and first column
  const int tr = tid / CLS, scol = (tid % CLS) * SPT;  // staging: input row of a pass, first column
  const uint32_t pitch = (uint32_t)s * sizeof(V);      // bytes of a row
  // row r of Xsub or Wout, from column q of the task's on
  auto xrow = [&](int r, int q) {
    return reinterpret_cast<V*>(reinterpret_cast<char*>(A.Xsub + c0 + q) + (uint64_t)(uint32_t)r * pitch);
  };
  auto wrow = [&](int r, int q) {
    return reinterpret_cast<V*>(reinterpret_cast<char*>(A.Wout + c0 + q) + (uint64_t)(uint32_t)r * pitch);
  };
  V* const own = A.Wout + T.row * s + c0;               // the front's own rows
  auto orow = [&](int r, int q) {
    return reinterpret_cast<V*>(reinterpret_cast<char*>(own + q) + (uint32_t)r * pitch);
  };

  // ring: stages of the warp's groups g0 + warp, + SW_NW, ... in order
  int ig = KS ? T.g0 : T.g0 + warp, il = 0, inb = 0, islot = 0;  // group, bytes of it left, bytes per full stage, slot
  const char* isrc = nullptr;
  const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
  auto open = [&]() {  // stage source of group ig
    if (ig < gend) {
      const int nrp = mf_group_rows(nout, ig);
      const int len = FWD ? min(k, MF_GR * (ig + 1)) : f - MF_GR * ig;
      isrc = reinterpret_cast<const char*>(A.M + T.m + (FWD ? mf_fwd_before(k, ig) : mf_bwd_before(f, ig)));
      inb = KC * nrp * (int)sizeof(V);
      il = len * nrp * (int)sizeof(V);
      if (KS) {
        isrc += warp * inb;
        il -= warp * inb;
      }
    }
  };
  auto issue = [&]() {
    if (il > 0) {
      const int bytes = min(inb, il);
      const uint32_t dst = ring_s + islot * BYTES;
#pragma unroll
      for (int o = 0; o < BYTES; o += 512)
        if (o + lane * 16 < bytes) cp_async16(dst + o + lane * 16, isrc + o + lane * 16);
      isrc += KS ? SW_NW * bytes : bytes;
      il -= KS ? SW_NW * bytes : bytes;
      if (!KS && il == 0) {
        ig += SW_NW;
        open();
      }
    }
    cp_async_commit();
    islot = islot + 1 == SW_NST ? 0 : islot + 1;
  };
  open();
#pragma unroll
  for (int i = 0; i < SW_NST - 1; ++i) issue();

  // input rows lb + u RPP + tr, u < N: their sources, then their values. The
  // backward rows are plain copies (FP32: cp.async, 16 columns of the 5 Hz
  // workload 4.28 -> 4.05 ms with the wider staging; FP64 gained nothing, as a
  // wait for them also waits for the ring); the forward ones are sums of up to
  // three rows and pass through registers, like one column's 8-byte rows.
  constexpr bool COPY = !FWD && L::F32 && SPT * sizeof(V) == 16;
  auto load_idx = [&](int lb, auto& xr, auto& cc) {
    constexpr int N = sizeof(xr) / sizeof(int);
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int l = lb + u * RPP + tr;
      xr[u] = -1;
      if (FWD) cc[u] = make_int2(-1, -1);
      if (l < hi) {
        if (FWD || l >= k) xr[u] = __ldg(A.rows + T.row + l);
        if (FWD && A.kids) cc[u] = __ldg(A.csrc + T.row + l);
      }
    }
  };
  auto load_val = [&](int lb, const auto& xr, const auto& cc, auto& v, auto& w0, auto& w1, V* dst) {
    constexpr int N = sizeof(xr) / sizeof(int);
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int l = lb + u * RPP + tr;
      if (l < hi) {
        const V* src = FWD || xr[u] >= 0 ? xrow(xr[u], scol) : orow(l, scol);
        if (COPY) {
          cp_async16((uint32_t)__cvta_generic_to_shared(dst + (u * RPP + tr) * S + scol), src);
        } else {
          ld_cols<SPT>(src, v[u]);
          if (FWD && A.kids) {
#pragma unroll
            for (int p = 0; p < SPT; ++p) w0[u][p] = w1[u][p] = c_zero<V>();
            if (cc[u].x >= 0) ld_cols<SPT>(wrow(cc[u].x, scol), w0[u]);
            if (cc[u].y >= 0) ld_cols<SPT>(wrow(cc[u].y, scol), w1[u]);
          }
        }
      }
    }
  };
  auto store_val = [&](V* dst, int lb, auto& v, const auto& w0, const auto& w1) {  // row lb at dst[0]
    constexpr int N = sizeof(v) / (SPT * sizeof(V));
    if (COPY) return;
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int l = u * RPP + tr;
      if (lb + l < hi) {
#pragma unroll
        for (int p = 0; p < SPT; ++p) {
          if (FWD && A.kids) v[u][p] = c_add(c_add(v[u][p], w0[u][p]), w1[u][p]);
          dst[l * S + scol + p] = v[u][p];
        }
      }
    }
  };

  // the whole input, or its first CH rows: NF passes at a time, the next sources ahead of the values
  int base = lo, end = STREAM ? min(lo + CH, hi) : hi;
  {
    constexpr int NF = STREAM ? U : ((FWD ? 32 : 128) / RPP > U ? (FWD ? 32 : 128) / RPP : U);
    int xr[NF];
    int2 cc[NF];
    load_idx(lo, xr, cc);
    if (!wait()) return false;
    for (int lb = lo; lb < end; lb += NF * RPP) {
      V v[NF][SPT], w0[NF][SPT], w1[NF][SPT];
      load_val(lb, xr, cc, v, w0, w1, bs + (lb - lo) * S);
      if (lb + NF * RPP < end) load_idx(lb + NF * RPP, xr, cc);
      store_val(bs + (lb - lo) * S, lb, v, w0, w1);
    }
  }
  if (COPY) {
    cp_async_commit();
    cp_async_wait<0>();
  }
  int xr[U];
  int2 cc[U];
  V v[U][SPT], w0[U][SPT], w1[U][SPT];
  if (STREAM) load_idx(end, xr, cc);

  SwAcc<V, S> acc, tot;
  acc.zero();
  if (!L::F32) tot.zero();
  int cg = KS ? T.g0 : T.g0 + warp, slot = 0, used = 0;  // group, ring slot being read, indices of it already used
  int ck = (FWD ? 0 : MF_GR * cg) + (KS ? warp * KC : 0);  // next reduction index of the group
  bool part = false;                         // `tot` holds the earlier chunks of the group
  // the lane's rows of the group: the first one, how many; where they go (backward), or the children's
  // updates that join them (forward)
  int r0 = 0, nv = 0, xo[FWD ? 1 : RPT];
  int2 ce[FWD ? RPT : 1];
  auto targets = [&]() {
    const int nrp = mf_group_rows(nout, min(cg, gend - 1)), rpt = SwAcc<V, S>::rows(nrp);
    r0 = MF_GR * cg + rg * rpt;
    nv = rg * rpt < nrp ? max(0, min(rpt, nout - r0)) : 0;
    if (cg >= gend) nv = 0;
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      if (FWD) {
        ce[i] = make_int2(-1, -1);
        if (A.kids && i < nv && r0 + i >= k) ce[i] = __ldg(A.csrc + T.row + r0 + i);
      } else {
        if (i < nv) xo[i] = __ldg(A.rows + T.row + r0 + i);
      }
    }
  };
  targets();
  V* buf = bs;
  while (true) {
    __syncthreads();
    const bool more = STREAM && end < hi;
    if (more) {
      load_val(end, xr, cc, v, w0, w1, buf == bs ? bs + CH * S : bs);  // joins the next ring stage's copies
      load_idx(end + CH, xr, cc);
    }
    while (cg < gend) {
      const int nrp = mf_group_rows(nout, cg);
      const int kfirst = FWD ? 0 : MF_GR * cg, klast = FWD ? min(k, MF_GR * (cg + 1)) : f;
      const int kstop = min(klast, end);
      const V* b = buf + col;
      while (ck < kstop) {
        if (!KS && (ck & (MF_CHUNK - 1)) == 0 && ck > kfirst) {  // a chunk is complete
          if (part || !L::F32)
            tot.add(acc);
          else
            tot = acc;
          acc.zero();
          part = true;
        }
        if (used == 0) {
          cp_async_wait<SW_NST - 2>();
          __syncwarp();
          issue();
        }
        const int n = min(min(KC - used, kstop - ck), KS ? KC : MF_CHUNK - (ck & (MF_CHUNK - 1)));
        acc.mac(ring + slot * STAGE + used * nrp, b + (ck - base) * S, n, nrp, rg, lane);
        ck += n;
        used += n;
        if (used == KC || ck == klast) {
          used = 0;
          if (KS) ck += (SW_NW - 1) * KC;
          slot = slot + 1 == SW_NST ? 0 : slot + 1;
        }
      }
      if (ck < klast || (KS && STREAM && end < hi)) break;  // goes on in the next rows
      if (KS) {  // the parts, in warp order, to warp 0
        SwAcc<V, S>* parts = reinterpret_cast<SwAcc<V, S>*>(smem);
        cp_async_wait<0>();
        __syncthreads();  // every warp has used its stages
        parts[tid] = acc;
        __syncthreads();
        if (warp == 0)
          for (int w = 1; w < SW_NW; ++w) acc.add(parts[32 * w + lane]);
        if (warp != 0) break;
      }
      // epilogue: all loads first, then the rows in order
      if (part) {
        tot.add(acc);
        acc = tot;
        if (!L::F32) tot.zero();
      }
      const int nst = L::SPLIT && (lane & 1) ? 0 : nv;  // rows the lane writes
      if (!FWD) {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
          V o[CPT];
#pragma unroll
          for (int q = 0; q < CPT; ++q) o[q] = acc.get(i, q);
          if (i < nst) st_cols<CPT>(xrow(xo[i], col), o);
        }
      } else {
        // rows at a time: all their loads, then their sums. FP64 adds zeros where there is no child: a
        // branch around each addition left its loads one behind the other (cube, 3 columns: 0.71 -> 0.64 ms)
        constexpr int NB = L::F32 ? (RPT < 2 ? 1 : 2) : RPT;
#pragma unroll
        for (int i0 = 0; i0 < RPT; i0 += NB) {
          V o[NB][CPT], x0[NB][CPT], x1[NB][CPT];
#pragma unroll
          for (int h = 0; h < NB; ++h) {
            if (!L::F32) {
#pragma unroll
              for (int q = 0; q < CPT; ++q) x0[h][q] = x1[h][q] = c_zero<V>();
            }
            if (ce[i0 + h].x >= 0) ld_cols<CPT>(wrow(ce[i0 + h].x, col), x0[h]);
            if (ce[i0 + h].y >= 0) ld_cols<CPT>(wrow(ce[i0 + h].y, col), x1[h]);
#pragma unroll
            for (int q = 0; q < CPT; ++q) o[h][q] = acc.get(i0 + h, q);
          }
          if (MF_GR * cg < k) {  // a group with pivot rows
#pragma unroll
            for (int h = 0; h < NB; ++h)
              if (i0 + h < nv && r0 + i0 + h < k) {
                const V di = __ldg(A.Dinv + T.d + r0 + i0 + h);
#pragma unroll
                for (int q = 0; q < CPT; ++q)
                  o[h][q] = part ? mul_dinv<true>(o[h][q], di) : mul_dinv<false>(o[h][q], di);
              }
          }
#pragma unroll
          for (int h = 0; h < NB; ++h) {
            if (!L::F32 || ce[i0 + h].x >= 0)
#pragma unroll
              for (int q = 0; q < CPT; ++q) o[h][q] = c_add(o[h][q], x0[h][q]);
            if (!L::F32 || ce[i0 + h].y >= 0)
#pragma unroll
              for (int q = 0; q < CPT; ++q) o[h][q] = c_add(o[h][q], x1[h][q]);
            if (i0 + h < nst) st_cols<CPT>(orow(r0 + i0 + h, col), o[h]);
          }
        }
      }
      acc.zero();
      part = false;
      cg += SW_NW;
      ck = FWD ? 0 : MF_GR * cg;
      if (!KS) targets();
    }
    if (!more) break;
    buf = buf == bs ? bs + CH * S : bs;
    store_val(buf, end, v, w0, w1);
    if (COPY) {
      cp_async_commit();
      cp_async_wait<0>();
    }
    base = end;
    end = min(end + CH, hi);
  }
  return true;
}

template <typename V, int S, bool FWD, bool STREAM, typename Wait>
__device__ __forceinline__ bool sweep_task(const SweepArgs<V>& A, const SweepTask& T, int c0, unsigned char* smem,
                                           Wait&& wait) {
  if (sizeof(V) == 16 && T.ng == 1) return sweep_task_t<V, S, FWD, STREAM, sizeof(V) == 16>(A, T, c0, smem, wait);
  return sweep_task_t<V, S, FWD, STREAM, false>(A, T, c0, smem, wait);
}

// CTAs per SM to leave registers for
template <typename V, int S, bool FWD, bool STREAM>
constexpr int sw_min_blocks() {
  return sizeof(V) == 16 ? 2 : (STREAM ? 4 : (S <= 2 ? 8 : (FWD && S == 16 ? 5 : 6)));
}

// One level of one sweep: blockIdx = task * (column blocks) + column block.
template <typename V, int S, bool FWD, bool STREAM>
__global__ void __launch_bounds__(SW_THREADS, sw_min_blocks<V, S, FWD, STREAM>()) k_sweep_level(SweepArgs<V> A, int ncb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_trigger();
  const int ti = blockIdx.x / ncb;
  const SweepTask T = A.tasks[ti];
  sweep_task<V, S, FWD, STREAM>(A, T, (blockIdx.x - ti * ncb) * S, smem_raw, [] {
    pdl_wait();
    return true;
  });
}

// ---------------------------------------------------------------------------
// One column in complex FP32, long reductions on a level of few groups: what
// counts is the chain of one row, its staged inputs, ring stages and
// multiply-adds in turn. A CTA takes one group, and its warps one chunk
// (MF_CHUNK reduction indices) each at a time; the chunks' sums meet in shared
// memory and are added in order, the order of the sums of the other forms.
// Against k_sweep_level, whose warps follow their group from end to end
// (quarter workload, one column, us a level): 109 tasks 39 -> 20, 193 30 -> 17,
// 264 35 -> 29, 480 24 -> 21, but 686 20 -> 22 and 1161 23 -> 36, where the
// level is wide enough and a CTA that stages its input for one group reads
// more; hence up to LG_TASKS, four CTAs of the wider form per SM. The
// application: 0.81 -> 0.60 ms (the earlier tiles, split at 128 indices: 0.67);
// 5 Hz workload 1.68 -> 1.66. Two ring stages: three and four take the CTAs
// their shared memory (0.61 -> 0.65 with every such level in this form).
// ---------------------------------------------------------------------------
constexpr int LG_KC = 32;                       // indices per ring stage (4 KB)
constexpr int LG_NST = 2;                       // ring stages per warp
constexpr unsigned LG_TASKS = 608;              // levels of fewer tasks
constexpr int LG_STAGE = LG_KC * MF_GR;         // entries per stage
constexpr int LG_ROWS = SW_NW * MF_CHUNK;       // input rows of a window, one chunk per warp
constexpr int LG_RPT = LG_ROWS / SW_THREADS;    // rows per thread
constexpr size_t LG_SMEM = (size_t)SW_NW * LG_NST * LG_STAGE * sizeof(float2) + 2 * LG_ROWS * sizeof(float2) +
                           2 * SW_NW * MF_GR * sizeof(float2);

// group g of the task; `wait` as in sweep_task_t
template <bool FWD, typename Wait>
__device__ __forceinline__ bool sweep_long(const SweepArgs<float2>& A, const SweepTask& T, int g, unsigned char* smem,
                                           Wait&& wait) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int k = T.k, f = T.f, nout = FWD ? f : k;
  const int lo = FWD ? 0 : MF_GR * g, hi = FWD ? min(k, MF_GR * (g + 1)) : f;
  const int c0 = lo / MF_CHUNK, cend = (hi + MF_CHUNK - 1) / MF_CHUNK;  // the group's chunks
  const int nrp = mf_group_rows(nout, g), r = MF_GR * g + tid;        // threads below MF_GR: an output row each
  float2* const ring = reinterpret_cast<float2*>(smem) + (size_t)warp * LG_NST * LG_STAGE;
  float2* const bs = reinterpret_cast<float2*>(smem) + (size_t)SW_NW * LG_NST * LG_STAGE;  // [2][LG_ROWS]
  float2* const parts = bs + 2 * LG_ROWS;                                                  // [2][warp][row]
  float2* const own = A.Wout + T.row;
  const float2* const M = A.M + T.m + (FWD ? mf_fwd_before(k, g) : mf_bwd_before(f, g));

  // ring: the stages of the warp's chunks c0 + warp, + SW_NW, ... in order; none spans two chunks
  const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
  int ic = c0 + warp, il = max(lo, ic * MF_CHUNK), islot = 0;
  auto issue = [&]() {
    if (ic < cend) {
      const int end = min(hi, (ic + 1) * MF_CHUNK), n = min(LG_KC, end - il), bytes = n * nrp * (int)sizeof(float2);
      const char* src = reinterpret_cast<const char*>(M + (int64_t)(il - lo) * nrp) + lane * 16;
      const uint32_t dst = ring_s + islot * (LG_STAGE * (int)sizeof(float2)) + lane * 16;
#pragma unroll
      for (int o = 0; o < LG_STAGE * (int)sizeof(float2); o += 512)
        if (o + lane * 16 < bytes) cp_async16(dst + o, src + o);
      il += n;
      if (il == end) {
        ic += SW_NW;
        il = ic * MF_CHUNK;
      }
    }
    cp_async_commit();
    islot = islot + 1 == LG_NST ? 0 : islot + 1;
  };
#pragma unroll
  for (int i = 0; i < LG_NST - 1; ++i) issue();

  // input rows of the window from chunk cw on: their sources, then their values
  int xr[LG_RPT];
  int2 cc[LG_RPT];
  float2 v[LG_RPT], w0[LG_RPT], w1[LG_RPT];
  auto load_idx = [&](int cw) {
#pragma unroll
    for (int i = 0; i < LG_RPT; ++i) {
      const int l = cw * MF_CHUNK + i * SW_THREADS + tid;
      xr[i] = -1;
      cc[i] = make_int2(-1, -1);
      if (l >= lo && l < hi) {
        if (FWD || l >= k) xr[i] = __ldg(A.rows + T.row + l);
        if (FWD && A.kids) cc[i] = __ldg(A.csrc + T.row + l);
      }
    }
  };
  auto load_val = [&](int cw) {
#pragma unroll
    for (int i = 0; i < LG_RPT; ++i) {
      const int l = cw * MF_CHUNK + i * SW_THREADS + tid;
      v[i] = w0[i] = w1[i] = make_float2(0.f, 0.f);
      if (l >= lo && l < hi) {
        v[i] = __ldcg(FWD || xr[i] >= 0 ? A.Xsub + xr[i] : own + l);
        if (cc[i].x >= 0) w0[i] = __ldcg(A.Wout + cc[i].x);
        if (cc[i].y >= 0) w1[i] = __ldcg(A.Wout + cc[i].y);
      }
    }
  };
  auto store_val = [&](float2* b) {
#pragma unroll
    for (int i = 0; i < LG_RPT; ++i)
      b[i * SW_THREADS + tid] = FWD && A.kids ? c_add(c_add(v[i], w0[i]), w1[i]) : v[i];
  };
  load_idx(c0);
  int xo = 0;
  int2 ce = make_int2(-1, -1);
  float2 di = make_float2(0.f, 0.f), tot = di;
  const bool out = tid < MF_GR && r < nout;
  if (out) {
    if (!FWD) xo = __ldg(A.rows + T.row + r);
    if (FWD && A.kids && r >= k) ce = __ldg(A.csrc + T.row + r);
    if (FWD && r < k) di = __ldg(A.Dinv + T.d + r);
  }
  if (!wait()) return false;

  load_val(c0);
  if (c0 + SW_NW < cend) load_idx(c0 + SW_NW);
  store_val(bs);
  auto add_parts = [&](int cw, int buf) {  // chunks cw..cw + 3, in order
    if (tid < MF_GR)
      for (int w = 0; w < SW_NW && cw + w < cend; ++w) {
        const float2 q = parts[(buf * SW_NW + w) * MF_GR + tid];
        tot = cw + w == c0 ? q : c_add(tot, q);
      }
  };
  int slot = 0, buf = 0;
  for (int cw = c0; cw < cend; cw += SW_NW, buf ^= 1) {
    __syncthreads();
    const bool more = cw + SW_NW < cend;
    if (more) {
      load_val(cw + SW_NW);
      if (cw + 2 * SW_NW < cend) load_idx(cw + 2 * SW_NW);
    }
    if (cw > c0) add_parts(cw - SW_NW, buf ^ 1);
    if (cw + warp < cend) {
      const int p = min(lane & 7, nrp / 2 - 1), end = min(hi, (cw + warp + 1) * MF_CHUNK);
      int ck = max(lo, (cw + warp) * MF_CHUNK);
      pair2 re = 0, im = 0;
      while (ck < end) {
        cp_async_wait<LG_NST - 2>();
        __syncwarp();
        issue();
        const int n = min(LG_KC, end - ck);
        const float4* a = reinterpret_cast<const float4*>(ring + slot * LG_STAGE) + p;
        const float2* b = bs + buf * LG_ROWS + (ck - cw * MF_CHUNK);
        auto step = [&](const float4 t, const float2 bv) {
          const pair2 ar = pk(t.x, t.y), ai = pk(t.z, t.w);
          const pair2 br = pk(bv.x, bv.x), bi = pk(bv.y, bv.y), nbi = pk(-bv.y, -bv.y);
          re = fma2(ar, br, fma2(ai, nbi, re));
          im = fma2(ar, bi, fma2(ai, br, im));
        };
        int kk = 0;
#pragma unroll 1
        for (; kk + 8 <= n; kk += 8) {
          float4 t[8];
          float2 bv[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            t[u] = a[(kk + u) * (nrp / 2)];
            bv[u] = b[kk + u];
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) step(t[u], bv[u]);
        }
#pragma unroll 1
        for (; kk < n; ++kk) step(a[kk * (nrp / 2)], b[kk]);
        ck += n;
        slot = slot + 1 == LG_NST ? 0 : slot + 1;
      }
      const float2 x = unpk(re), y = unpk(im);
      if (lane < nrp / 2)
        reinterpret_cast<float4*>(parts)[((buf * SW_NW + warp) * MF_GR) / 2 + lane] = make_float4(x.x, y.x, x.y, y.y);
    }
    if (more) store_val(bs + (buf ^ 1) * LG_ROWS);
  }
  __syncthreads();
  if (cend > c0) {
    const int nw = (cend - c0 + SW_NW - 1) / SW_NW;
    add_parts(c0 + (nw - 1) * SW_NW, (nw - 1) & 1);
  }
  if (out) {
    if (!FWD) {
      A.Xsub[xo] = tot;
    } else {
      float2 x0 = make_float2(0.f, 0.f), x1 = x0;
      if (ce.x >= 0) x0 = __ldcg(A.Wout + ce.x);
      if (ce.y >= 0) x1 = __ldcg(A.Wout + ce.y);
      if (r < k) tot = cend > 1 ? mul_dinv<true>(tot, di) : mul_dinv<false>(tot, di);
      if (ce.x >= 0) tot = c_add(tot, x0);
      if (ce.y >= 0) tot = c_add(tot, x1);
      own[r] = tot;
    }
  }
  return true;
}

// One level of one sweep in that form: blockIdx = task * SW_NW + group of the task.
template <bool FWD>
__global__ void __launch_bounds__(SW_THREADS, 5) k_sweep_long(SweepArgs<float2> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_trigger();
  const SweepTask T = A.tasks[blockIdx.x / SW_NW];
  const int q = blockIdx.x % SW_NW;
  if (q >= T.ng) return;  // the task's first CTA waits for the previous launch
  sweep_long<FWD>(A, T, T.g0 + q, smem_raw, [] {
    pdl_wait();
    return true;
  });
}

// ---------------------------------------------------------------------------
// Persistent sweeps (option persistent_sweeps): one launch per direction over
// every level. Resident CTAs take the tasks in level order through a ticket
// counter (the forward sweep from the leaves up, the backward sweep from the
// roots down). Before it reads its inputs, a CTA waits until they are final:
// forward, every child front with rows has finished; backward, the nearest
// ancestor with pivots has (so all the ancestors' pivots are final). A front
// has finished when all its tasks have; then (forward) it counts itself into
// its parent. Every dependency has a smaller ticket, and a ticket is only
// taken by a running CTA, so the smallest unfinished ticket can always
// proceed. Waits are bounded by the global timer; a timeout sets *err and the
// CTA stops taking tasks (the sweep's result is then invalid and reported).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t sw_clock_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ int sw_load(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// wait until *p >= target; false after about two seconds
__device__ __forceinline__ bool sw_wait(const int* p, int target) {
  if (sw_load(p) >= target) return true;
  const uint64_t t0 = sw_clock_ns();
  while (sw_load(p) < target) {
    __nanosleep(200);
    if (sw_clock_ns() - t0 > 2000000000ull) return false;
  }
  return true;
}

template <typename V, int S, bool FWD>
__global__ void __launch_bounds__(SW_THREADS, sw_min_blocks<V, S, FWD, true>()) k_sweep_all(
    SweepArgs<V> A, int ncb, int ntasks, const int* __restrict__ front_tasks, const int* __restrict__ dep,
    const int* __restrict__ nchild, int* __restrict__ cnt, int nfronts, int* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_ticket, s_ok;
  int* front_done = cnt + 1;
  int* child_ready = front_done + nfronts;
  const int total = ntasks * ncb;
  while (true) {
    if (threadIdx.x == 0) s_ticket = atomicAdd(cnt, 1);
    __syncthreads();
    const int tk = s_ticket;
    if (tk >= total) break;
    const int ti = tk / ncb;
    const SweepTask T = A.tasks[ti];
    const int g = T.front;
    const bool ok = sweep_task<V, S, FWD, true>(A, T, (tk - ti * ncb) * S, smem_raw, [&] {
      if (threadIdx.x == 0) {
        bool o = true;
        if (FWD)
          o = sw_wait(child_ready + g, nchild[g]);
        else if (dep[g] >= 0)
          o = sw_wait(front_done + dep[g], front_tasks[dep[g]] * ncb);
        if (!o) atomicExch(err, 1);
        s_ok = o;
      }
      __syncthreads();
      return s_ok != 0;
    });
    if (!ok) {
      cp_async_wait<0>();  // the ring's copies land before the CTA exits
      break;
    }
    __threadfence();
    __syncthreads();  // every write of the task is issued; s_ticket may be overwritten
    if (threadIdx.x == 0 && atomicAdd(front_done + g, 1) == front_tasks[g] * ncb - 1 && FWD && dep[g] >= 0) {
      __threadfence();
      atomicAdd(child_ready + dep[g], 1);
    }
  }
}

template <typename V, int S, bool FWD, bool STREAM>
size_t sw_smem(int rows) {
  return (size_t)SW_NW * SW_NST * SwV<V, FWD, STREAM>::BYTES + (size_t)rows * S * sizeof(V);
}

// The tasks of level l. A level whose longest reduction fits stages its
// inputs whole.
template <typename V, int S, bool FWD>
void launch_level(const DevMF& mf, SweepArgs<V>& A, int l, cudaStream_t st) {
  const int* ptr = FWD ? mf.ftask_ptr_h : mf.btask_ptr_h;
  const int ncb = A.s / S, rows = (FWD ? mf.fbrows_h : mf.bbrows_h)[l];
  const unsigned grid = (unsigned)(ptr[l + 1] - ptr[l]) * ncb;
  A.tasks = (FWD ? mf.ftasks : mf.btasks) + ptr[l];
  if constexpr (sizeof(V) == 8 && S == 1)
    if (rows > MF_RES && grid < LG_TASKS) {
      launch_k(true, k_sweep_long<FWD>, grid * SW_NW, SW_THREADS, LG_SMEM, st, A);
      return;
    }
  if (rows <= MF_RES)
    launch_k(true, k_sweep_level<V, S, FWD, false>, grid, SW_THREADS, sw_smem<V, S, FWD, false>(rows), st, A, ncb);
  else
    launch_k(true, k_sweep_level<V, S, FWD, true>, grid, SW_THREADS, sw_smem<V, S, FWD, true>(2 * SwS<V, S, FWD>::CH), st, A,
             ncb);
}

// One level with the widest column block that still gives the SMs two warps
// per scheduler (1216), down to 4 columns: narrower blocks read the factor
// more often (from L2) but shorten the chain of a level of few, long rows.
// Against always the widest: two-level at 5 Hz, 16 columns, 17.6 ms to 18.5;
// quarter, 5 columns, 1.01 to 1.05; FP64, 16 columns, 26.4 to 27.2; elsewhere equal.
template <typename V, bool FWD>
void sweep_level(const DevMF& mf, SweepArgs<V>& A, int l, cudaStream_t st) {
  const int* ptr = FWD ? mf.ftask_ptr_h : mf.btask_ptr_h;
  if (ptr[l + 1] == ptr[l]) return;
  A.M = (const V*)(FWD ? mf.M : mf.MT);
  A.kids = l > 0;  // level 0 holds the leaves
  const int64_t groups = (FWD ? mf.fgroups_h : mf.bgroups_h)[l];
  int w = A.s % 16 == 0 ? 16 : (A.s % 8 == 0 ? 8 : A.s);
  while (w > 4 && groups * (A.s / w) < 1216) w /= 2;
  switch (w) {
    case 1: launch_level<V, 1, FWD>(mf, A, l, st); break;
    case 2: launch_level<V, 2, FWD>(mf, A, l, st); break;
    case 4: launch_level<V, 4, FWD>(mf, A, l, st); break;
    case 8: launch_level<V, 8, FWD>(mf, A, l, st); break;
    default: launch_level<V, 16, FWD>(mf, A, l, st);
  }
}

template <typename V, int S, bool FWD>
void sweep_all(const DevMF& mf, SweepArgs<V>& A, cudaStream_t st) {
  const int ncb = A.s / S;
  const int nt = (FWD ? mf.ftask_ptr_h : mf.btask_ptr_h)[mf.nlevels];
  if (nt == 0) return;
  const size_t shm = sw_smem<V, S, FWD, true>(2 * SwS<V, S, FWD>::CH);
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sweep_all<V, S, FWD>, SW_THREADS, shm);
  A.kids = 1;
  A.tasks = FWD ? mf.ftasks : mf.btasks_top;
  A.M = (const V*)(FWD ? mf.M : mf.MT);
  cudaMemsetAsync(mf.cnt, 0, (size_t)(1 + 2 * mf.nfronts) * sizeof(int), st);
  launch_k(false, k_sweep_all<V, S, FWD>, (unsigned)std::min<int64_t>((int64_t)per * sms, (int64_t)nt * ncb),
           SW_THREADS, shm, st, A, ncb, nt, (const int*)(FWD ? mf.front_ftasks : mf.front_btasks),
           (const int*)(FWD ? mf.parent : mf.bdep), (const int*)mf.nchild, mf.cnt, (int)mf.nfronts, mf.sw_err);
}

template <typename V>
void solve_v(DevMF& mf, V* Xsub, int cols, cudaStream_t st) {
  SweepArgs<V> A;
  A.rows = mf.rows;
  A.csrc = mf.csrc;
  A.Dinv = (const V*)mf.Dinv;
  A.Xsub = Xsub;
  A.Wout = (V*)mf.Wout;
  A.s = cols;
  // One FP32 column on a tree that fills the SMs goes level by level in either
  // case: the persistent form keeps the chains that k_sweep_long cuts (cube of
  // 6^3 cells 0.141 ms to 0.110, quarter workload 0.84 to 0.61, 5 Hz 2.65 to
  // 1.74). Trees of fewer tasks gain from the launches saved (two-level, cube,
  // with its coarse level of 1000 dofs level by level 1.87 ms, persistent 1.80).
  if (mf.persistent && !(sizeof(V) == 8 && cols == 1 && mf.ftask_ptr_h[mf.nlevels] >= (int)LG_TASKS)) {
    auto both = [&](auto w) {
      sweep_all<V, decltype(w)::value, true>(mf, A, st);
      sweep_all<V, decltype(w)::value, false>(mf, A, st);
    };
    if (cols == 1)
      both(std::integral_constant<int, 1>());
    else if (cols == 2)
      both(std::integral_constant<int, 2>());
    else if (cols == 4)
      both(std::integral_constant<int, 4>());
    else if (cols % 16)
      both(std::integral_constant<int, 8>());
    else
      both(std::integral_constant<int, 16>());
    return;
  }
  for (int l = 0; l < mf.nlevels; ++l) sweep_level<V, true>(mf, A, l, st);
  for (int l = mf.nlevels - 1; l >= 0; --l) sweep_level<V, false>(mf, A, l, st);
}

template <typename V, int S, bool FWD>
void attrs_sf() {
  const int whole = (int)sw_smem<V, S, FWD, false>(MF_RES), stream = (int)sw_smem<V, S, FWD, true>(2 * SwS<V, S, FWD>::CH);
  cudaFuncSetAttribute(k_sweep_level<V, S, FWD, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, whole);
  cudaFuncSetAttribute(k_sweep_level<V, S, FWD, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, stream);
  cudaFuncSetAttribute(k_sweep_all<V, S, FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, stream);
  if constexpr (sizeof(V) == 8 && S == 1)
    cudaFuncSetAttribute(k_sweep_long<FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LG_SMEM);
}
template <typename V, int S>
void attrs_s() {
  attrs_sf<V, S, true>();
  attrs_sf<V, S, false>();
}

}  // namespace

// Row length of the sub-vector and front vectors of a block of s columns: the
// sweeps work on whole column blocks of 1, 2, 4, 8 or 16 (the columns past s
// are computed and never read).
int sweep_cols(int s) { return s <= 2 ? s : (s <= 4 ? 4 : (s <= 8 ? 8 : (s <= 16 ? 16 : (s + 7) / 8 * 8))); }

// Opt the sweep kernels into their dynamic shared memory, outside any stream capture.
void sweep_attrs(bool fp32) {
  if (fp32) {
    attrs_s<float2, 1>();
    attrs_s<float2, 2>();
    attrs_s<float2, 4>();
    attrs_s<float2, 8>();
    attrs_s<float2, 16>();
  } else {
    attrs_s<double2, 1>();
    attrs_s<double2, 2>();
    attrs_s<double2, 4>();
    attrs_s<double2, 8>();
    attrs_s<double2, 16>();
  }
}

void sweep_solve(DevMF& mf, void* Xsub, int cols, cudaStream_t st) {
  if (mf.fp32)
    solve_v<float2>(mf, (float2*)Xsub, cols, st);
  else
    solve_v<double2>(mf, (double2*)Xsub, cols, st);
}

}  // namespace hz
