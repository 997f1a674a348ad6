// Local solves of the tensor-core form (option tensor_cores), and the entry
// points of the factorisation and the solve.
//
// With tensor_cores = 1, blocks of 9-16 columns run the front sweeps
// (sweep.cu has the products) as 128 x 128 tiles, split along the reduction:
// the larger tiles as tcgen05 MMAs, the others as SIMT tiles beside them, and
// a fixed-order sum of the tiles' partial results. Every other width, and
// every width without the option, runs the sweeps of sweep.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <utility>

#include "kernels.cuh"

#include "cplx.cuh"

namespace hz {

static void tile_attrs();
static void tc_pack_all(DevMF& mf, cudaStream_t st);
void mf_factor_fronts(DevMF& mf, double tau_abs, cudaStream_t st);  // factor.cu

// Numeric factorisation and partitioned inverse (factor.cu), then the
// sweep kernels' attributes and the tensor-core tile packing.
void mf_factor(DevMF& mf, double tau_abs, cudaStream_t st) {
  sweep_attrs(mf.fp32 != 0);
  if (mf.tc) tile_attrs();
  mf_factor_fronts(mf, tau_abs, st);
  // tensor-core tiles: pack their factor blocks from X_t (forward) and X_t^T (backward)
  if (mf.tc && mf.fp32) tc_pack_all(mf, st);
}

bool mf_tc_usable(const DevMF& mf, int s) { return mf.tc && mf.fp32 && s > 8 && s <= 16; }

// ---------------------------------------------------------------------------
// SIMT tiles beside the tensor-core tiles (complex FP32, 16 columns)
// ---------------------------------------------------------------------------
constexpr int MF_TILE = 128;  // output rows per tile (MF_TILE_ROWS on the host)
constexpr int MF_TK = 128;    // reduction length per tile (MF_TILE_K on the host)
constexpr int TS = 16;        // columns

// One tile: MF_TILE output rows x MF_TK reduction indices of
//   forward : t = X_t b_P;  backward: x = X_t^T [y_P; x_U].
// A row block covered by one tile (slot < 0) applies the epilogue directly;
// otherwise the tile writes a partial result to its slot of P and the row
// block's partials are summed in a fixed order by k_mf_reduce. Epilogue:
//   forward : rows r < k -> y = t / D (kept in Wout for the backward sweep);
//             rows r >= k -> parent update c_U + t (Wout), c_U = the children's
//             update vectors landing on the row
//   backward: x at the pivot rows of the sub-vector
// TPR threads share each output row, each keeping TS / TPR of the columns as
// register accumulators; the tile's input rows are staged once in shared
// memory and each thread streams its row of the factor tile, MF_UNROLL
// reduction indices ahead. Short levels (fewer than MF_SHORT_LEVEL tiles) run
// four threads per row; long levels whose tiles all have at most MF_HALF
// output rows run half-height tiles with two threads per row; the others one.
constexpr int MF_UNROLL = 8;
constexpr int MF_SHORT_LEVEL = 1536;
constexpr int MF_HALF = 64;
// 1024 resident threads per SM with several threads per row, 6 half-height
// tiles of 128 threads, 5 blocks of 128 with one thread per row
template <int TPR, int ROWS>
__host__ __device__ constexpr int tile_min_blocks() {
  return ROWS < MF_TILE ? 6 : (TPR > 1 ? 1024 / (MF_TILE * TPR) : 5);
}

template <bool FWD, int TPR, int ROWS>
__global__ void __launch_bounds__(ROWS* TPR, tile_min_blocks<TPR, ROWS>()) k_mf_tile(
    const int4* __restrict__ tiles, const int* __restrict__ kk, const int* __restrict__ ff,
    const int64_t* __restrict__ rowoff, const int64_t* __restrict__ Moff, const float2* __restrict__ M,
    const int* __restrict__ rows, const int2* __restrict__ csrc, const int64_t* __restrict__ Doff,
    const float2* __restrict__ Dinv, float2* __restrict__ Xsub, float2* __restrict__ Wout, float2* __restrict__ P,
    int s) {
  using V = float2;
  static_assert(TS % TPR == 0, "columns split evenly over the threads of a row");
  static_assert(ROWS <= MF_TILE, "a tile computes at most MF_TILE output rows");
  constexpr int CPT = TS / TPR;  // columns per thread
  __shared__ V bs[MF_TK][TS];
  const int4 tile = tiles[blockIdx.x];
  const int t = tile.x, r0 = tile.y, c0 = tile.z, slot = tile.w;
  const int f = ff[t], k = kk[t];
  const int nout = FWD ? f : k;
  const int kend = FWD ? ((r0 < k) ? min(k, r0 + MF_TILE) : k) : f;
  const int kbeg = FWD ? c0 : max(c0, r0);  // X_t^T is zero left of the diagonal of its pivot block
  const int kstop = min(kend, c0 + MF_TK);
  const int64_t ro = rowoff[t];
  const int tid = threadIdx.x;
  const int row = tid / TPR, cb = (tid % TPR) * CPT;  // output row of the tile, first column
  const int lmax = max(0, kstop - kbeg);
  const int rr = r0 + row;
  const bool act = rr < nout;
  // the row's group and its stored reduction range [l0, l1), relative to kbeg
  const int grp = rr / MF_GR, rl = rr % MF_GR;
  const int l0 = FWD ? 0 : max(0, MF_GR * grp - kbeg);
  const int l1 = act ? (FWD ? min(lmax, min(k, MF_GR * (grp + 1)) - kbeg) : lmax) : 0;
  const int ld = act ? mf_group_rows(nout, grp) : 0;
  const int i0 = kbeg - (FWD ? 0 : MF_GR * grp);  // index inside the group of kbeg
  const V* mg = M + Moff[t] + (act ? (FWD ? mf_fwd_before(k, grp) : mf_bwd_before(f, grp)) : 0);
  // the first factor entries are read while the input rows are staged
  V m0[MF_UNROLL];
#pragma unroll
  for (int u = 0; u < MF_UNROLL; ++u) m0[u] = u >= l0 && u < l1 ? mf_get(mg, ld, i0 + u, rl) : c_zero<V>();
  for (int l = row; l < lmax; l += ROWS) {
    const int64_t R = ro + kbeg + l;
    const int local = kbeg + l;
    V v[CPT];
    const V* src = (FWD || local >= k) ? Xsub + (int64_t)rows[R] * s : Wout + R * s;
#pragma unroll
    for (int q = 0; q < CPT; ++q) v[q] = cb + q < s ? src[cb + q] : c_zero<V>();
    if (FWD) {
      const int2 cc = csrc[R];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int cr = h ? cc.y : cc.x;
        if (cr < 0) continue;
        const V* w = Wout + (int64_t)cr * s;
#pragma unroll
        for (int q = 0; q < CPT; ++q)
          if (cb + q < s) v[q] = c_add(v[q], w[cb + q]);
      }
    }
#pragma unroll
    for (int q = 0; q < CPT; ++q) bs[l][cb + q] = v[q];
  }
  __syncthreads();
  V acc[CPT];
#pragma unroll
  for (int q = 0; q < CPT; ++q) acc[q] = c_zero<V>();
  // software pipeline: the next MF_UNROLL factor entries are in flight while the current ones are used
  int j = 0;
  while (j < l1) {
    const int jn = j + MF_UNROLL;
    V m1[MF_UNROLL];
#pragma unroll
    for (int u = 0; u < MF_UNROLL; ++u)
      m1[u] = jn + u >= l0 && jn + u < l1 ? mf_get(mg, ld, i0 + jn + u, rl) : c_zero<V>();
#pragma unroll
    for (int u = 0; u < MF_UNROLL; ++u)
      if (j + u < l1)
#pragma unroll
        for (int q = 0; q < CPT; ++q) acc[q] = c_fma(m0[u], bs[j + u][cb + q], acc[q]);
#pragma unroll
    for (int u = 0; u < MF_UNROLL; ++u) m0[u] = m1[u];
    j = jn;
  }
  if (slot >= 0) {
    V* out = P + ((int64_t)slot * MF_TILE + row) * s;
#pragma unroll
    for (int q = 0; q < CPT; ++q)
      if (cb + q < s) out[cb + q] = acc[q];
    return;
  }
  if (!act) return;
  const int64_t Rg = ro + rr;
  if (FWD) {
    if (rr < k) {
      const V di = Dinv[Doff[t] + rr];
#pragma unroll
      for (int q = 0; q < CPT; ++q)
        if (cb + q < s) Wout[Rg * s + cb + q] = c_mul(acc[q], di);
    } else {
      // parent update: the children's update vectors landing on this row
      const int2 cc = csrc[Rg];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int cr = h ? cc.y : cc.x;
        if (cr < 0) continue;
        const V* w = Wout + (int64_t)cr * s;
#pragma unroll
        for (int q = 0; q < CPT; ++q)
          if (cb + q < s) acc[q] = c_add(acc[q], w[cb + q]);
      }
#pragma unroll
      for (int q = 0; q < CPT; ++q)
        if (cb + q < s) Wout[Rg * s + cb + q] = acc[q];
    }
  } else {
    V* xo = Xsub + (int64_t)rows[Rg] * s;
#pragma unroll
    for (int q = 0; q < CPT; ++q)
      if (cb + q < s) xo[cb + q] = acc[q];
  }
}

// Epilogues of the split row blocks of one level (rb = front, first row,
// tiles, first slot), one thread per (row, column): the partial tiles are
// summed in slot order, then as in the tile's own epilogue.
template <bool FWD>
__global__ void k_mf_reduce(const int4* __restrict__ rblocks, int nrb, const int* __restrict__ kk,
                            const int* __restrict__ ff, const int64_t* __restrict__ rowoff,
                            const int64_t* __restrict__ Doff, const int* __restrict__ rows,
                            const int2* __restrict__ csrc, const float2* __restrict__ Dinv, float2* __restrict__ Wout,
                            const float2* __restrict__ P, float2* __restrict__ Xsub, int s) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t per = (int64_t)MF_TILE * s;
  if (g >= nrb * per) return;
  const int i = (int)((g % per) / s), c = (int)(g % s);
  const int4 rb = rblocks[g / per];
  const int t = rb.x, r = rb.y + i;
  const int k = kk[t];
  if (r >= (FWD ? ff[t] : k)) return;
  float2 acc = make_float2(0.f, 0.f);
  for (int q = 0; q < rb.z; ++q) acc = c_add(acc, P[((int64_t)(rb.w + q) * MF_TILE + i) * s + c]);
  const int64_t R = rowoff[t] + r;
  if (FWD) {
    if (r < k) {
      Wout[R * s + c] = c_mul(acc, Dinv[Doff[t] + r]);
    } else {
      const int2 cc = csrc[R];
      if (cc.x >= 0) acc = c_add(acc, Wout[(int64_t)cc.x * s + c]);
      if (cc.y >= 0) acc = c_add(acc, Wout[(int64_t)cc.y * s + c]);
      Wout[R * s + c] = acc;
    }
  } else {
    Xsub[(int64_t)rows[R] * s + c] = acc;
  }
}

// ---------------------------------------------------------------------------
// Tensor-core tiles (complex FP32 form): the same tile product on tcgen05,
// with FP32 accuracy from a three-term TF32 split (Markidis et al. 2018:
// a = a_hi + a_lo with a_hi = a rounded to TF32, a_lo = a - a_hi also in
// TF32; a b ~ a_hi b_hi + a_hi b_lo + a_lo b_hi, the dropped a_lo b_lo being
// ~2^-22 relative).
//
// The tile's factor block is packed once, after the factorisation, as
// 16-column chunks; each chunk holds a real and an imaginary plane of
// nr8 = roundup(rows, 8) rows x 16 reduction indices in FP32, in the
// K-major layout of 8-row x 16-byte core matrices (a row group's 4 core
// matrices are adjacent, row groups 512 bytes apart), reduction indices past
// the tile's end zero. A chunk is two contiguous copies (cp.async.bulk) into
// a ring of shared-memory stages; once it has landed, the CTA truncates it
// in place to its TF32 high part and writes the low part beside it. The input
// rows are staged once per tile as N x 128 operands, N = 2S, in high and low
// parts: B1 = [Re b | Im b] and B2 = [-Im b | Re b], so that
//   D = Re(M) B1^T + Im(M) B2^T = [Re(M b) | Im(M b)]
// accumulates in TMEM (128 lanes = output rows, N columns, FP32). Thread 0
// issues the MMAs (M = 128, N = 2S, K = 8 per instruction, 6 per 8 reduction
// indices) and commits them to the ring's barriers. Every wait is bounded by
// the global timer; a timeout sets *err, skips the epilogue, and the CTA
// waits (bounded again) for its copies in flight and its MMAs before it
// frees its TMEM and exits. Rows past the tile's end hold stale shared
// memory; their outputs are never written.
// ---------------------------------------------------------------------------
constexpr int TC_PLANE = 8192;              // one plane of a 128-row chunk in shared memory
constexpr int TC_STAGE = 2 * TC_PLANE;      // a chunk (real + imaginary plane)
constexpr int TC_SBO_A = 4 * 128;           // row-group stride of a 16-column chunk
constexpr int TC_SBO_B = (MF_TK / 4) * 128; // row-group stride of an N x 128 operand

__device__ __forceinline__ uint32_t tc_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// shared-memory matrix descriptor: no swizzle, K-major, descriptor version 1
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
__device__ __forceinline__ uint64_t tc_clock_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// wait for phase `parity` of an mbarrier, giving up after about half a second
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity) {
  uint32_t done = 0;
  const uint64_t t0 = tc_clock_ns();
  while (!done) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (!done && tc_clock_ns() - t0 > 500000000ull) return false;
  }
  return true;
}
// TF32 value of x by truncation of the 13 low mantissa bits: the high part
// of the split, exactly representable in TF32, with x - hi exact in FP32
__device__ __forceinline__ float tc_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }
// byte offset of element (row, col) in a K-major core-matrix tile whose row
// groups are sbo bytes apart
__device__ __forceinline__ int tc_off(int row, int col, int sbo) {
  return (row >> 3) * sbo + (col >> 2) * 128 + (row & 7) * 16 + (col & 3) * 4;
}

// tile geometry shared by the packer and the kernel
struct TcGeom {
  int t, r0, slot, f, k, nout, kbeg, kstop, nr, nr8, nk, nch;
};
template <bool FWD>
__device__ __forceinline__ TcGeom tc_geom(int4 tile, const int* kk, const int* ff) {
  TcGeom g;
  g.t = tile.x;
  g.r0 = tile.y;
  g.slot = tile.w;
  g.f = ff[g.t];
  g.k = kk[g.t];
  g.nout = FWD ? g.f : g.k;
  const int kend = FWD ? ((g.r0 < g.k) ? min(g.k, g.r0 + MF_TILE) : g.k) : g.f;
  g.kbeg = FWD ? tile.z : max(tile.z, g.r0);
  g.kstop = min(kend, tile.z + MF_TK);
  g.nr = min(MF_TILE, g.nout - g.r0);
  g.nr8 = (g.nr + 7) & ~7;
  g.nk = g.kstop - g.kbeg;
  g.nch = (g.nk + 15) / 16;
  return g;
}

// Pack the factor blocks of the tensor-core tiles (after the factorisation), FP32.
template <bool FWD>
__global__ void k_tc_pack(const int4* __restrict__ tiles, const int64_t* __restrict__ off, const int* __restrict__ kk,
                          const int* __restrict__ ff, const int64_t* __restrict__ Moff, const float2* __restrict__ M,
                          unsigned char* __restrict__ TC) {
  const TcGeom g = tc_geom<FWD>(tiles[blockIdx.x], kk, ff);
  const float2* Mt = M + Moff[g.t];
  unsigned char* base = TC + off[blockIdx.x];
  const int plane = g.nr8 * 64;
  const int64_t total = (int64_t)g.nch * 16 * g.nr8;
  for (int64_t i = threadIdx.x; i < total; i += blockDim.x) {
    const int m = (int)(i % g.nr8);
    const int kc = (int)((i / g.nr8) % 16);
    const int q = (int)(i / ((int64_t)g.nr8 * 16));
    const int col = g.kbeg + q * 16 + kc;
    float2 v = make_float2(0.f, 0.f);
    if (m < g.nr && col < g.kstop) {
      const int r = g.r0 + m;
      const int gr = r / MF_GR;
      if (FWD && col / MF_GR <= gr)
        v = mf_get(Mt + mf_fwd_before(g.k, gr), mf_group_rows(g.f, gr), col, r - MF_GR * gr);
      if (!FWD && gr <= col / MF_GR)
        v = mf_get(Mt + mf_bwd_before(g.f, gr), mf_group_rows(g.k, gr), col - MF_GR * gr, r - MF_GR * gr);
    }
    unsigned char* ch = base + (int64_t)q * 2 * plane;
    const int o = tc_off(m, kc, TC_SBO_A);
    *reinterpret_cast<float*>(ch + o) = v.x;
    *reinterpret_cast<float*>(ch + plane + o) = v.y;
  }
}

static void tc_pack_all(DevMF& mf, cudaStream_t st) {
  if (mf.ftc_n)
    { k_tc_pack<true><<<(unsigned)mf.ftc_n, 256, 0, st>>>(mf.ftiles_tc, mf.ftc_off, mf.k, mf.f, mf.Moff,
                                                         (const float2*)mf.M, mf.TC); count_launch(); }
  if (mf.btc_n)
    { k_tc_pack<false><<<(unsigned)mf.btc_n, 256, 0, st>>>(mf.btiles_tc, mf.btc_off, mf.k, mf.f, mf.MToff,
                                                          (const float2*)mf.MT, mf.TC); count_launch(); }
}

// shared memory of the tensor-core tile (96 KB, two CTAs per SM): the input
// operand B = [Re b | Im b] (N x 128) in high and low parts, a ring of
// TC_NRAW raw factor chunks and one working chunk (high part | low part)
// that the MMAs read
constexpr int TC_NRAW = 2;
template <int S>
static constexpr size_t tc_smem_bytes() {
  return 2 * (size_t)(2 * S) * MF_TK * 4 + (size_t)TC_NRAW * TC_STAGE + 2 * (size_t)TC_STAGE;
}

__device__ __forceinline__ void tc_mma(uint32_t taddr, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(taddr),
      "l"(da), "l"(db), "r"(idesc), "r"(acc));
}

// Complex product on real MMAs: D1 = Re(M) B and D2 = Im(M) B accumulate in
// two TMEM blocks of N = 2S columns; the epilogue forms
//   Re(M b) = D1[:, 0:S] - D2[:, S:2S],  Im(M b) = D1[:, S:2S] + D2[:, 0:S].
// Chunk pipeline (128 threads): thread 0 keeps TC_NRAW raw chunks in flight;
// every thread waits for chunk q and for the MMAs of chunk q - 1 (which read
// the working buffer), splits the raw chunk into its high and low parts in
// the working buffer, and after a CTA barrier (which also frees the raw stage
// for the copy of chunk q + TC_NRAW) thread 0 issues the six MMAs per 8
// reduction indices and commits them to the working buffer's barrier.
template <int S, bool FWD>
__global__ void __launch_bounds__(MF_TILE) k_mf_tile_tc(
    const int4* __restrict__ tiles, const int64_t* __restrict__ tcoff, const unsigned char* __restrict__ TC,
    const int* __restrict__ kk, const int* __restrict__ ff, const int64_t* __restrict__ rowoff,
    const int* __restrict__ rows, const int2* __restrict__ csrc, const int64_t* __restrict__ Doff,
    const float2* __restrict__ Dinv, float2* __restrict__ Xsub, float2* __restrict__ Wout, float2* __restrict__ P, int s,
    int* __restrict__ err) {
  static_assert(S == 16, "tensor-core tiles are built for blocks of 16 columns");
  constexpr int N = 2 * S;
  constexpr int BT = N * MF_TK * 4;
  constexpr uint32_t NCOL = 2 * N;  // D1 and D2
  extern __shared__ __align__(1024) unsigned char smem_tc[];
  unsigned char* sBh = smem_tc;
  unsigned char* sBl = smem_tc + BT;
  unsigned char* raw = smem_tc + 2 * BT;            // TC_NRAW x TC_STAGE
  unsigned char* wh = raw + TC_NRAW * TC_STAGE;     // working chunk, high part (real plane, imaginary plane)
  unsigned char* wl = wh + TC_STAGE;                // low part
  __shared__ __align__(8) uint64_t full[TC_NRAW], freeb, done;
  __shared__ uint32_t tslot;
  __shared__ int s_ok;
  const int tid = threadIdx.x, warp = tid >> 5;
  const TcGeom g = tc_geom<FWD>(tiles[blockIdx.x], kk, ff);
  const unsigned char* src = TC + tcoff[blockIdx.x];
  const uint32_t plane = (uint32_t)g.nr8 * 64, cbytes = 2 * plane;
  if (tid == 0) {
    for (int i = 0; i < TC_NRAW; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&full[i])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&freeb)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(&done)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_ok = 1;
  }
  __syncthreads();
  int issued = 0;  // thread 0: chunks whose copies were issued
  auto load_chunk = [&](int q) {  // thread 0: chunk q into raw stage q % TC_NRAW
    const uint32_t bar = tc_smem(&full[q % TC_NRAW]);
    const uint32_t dst = tc_smem(raw + (q % TC_NRAW) * TC_STAGE);
    const unsigned char* c = src + (int64_t)q * cbytes;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(cbytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(c), "r"(plane), "r"(bar)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     dst + TC_PLANE),
                 "l"(c + plane), "r"(plane), "r"(bar)
                 : "memory");
    issued = q + 1;
  };
  if (tid == 0)
    for (int q = 0; q < min(TC_NRAW, g.nch); ++q) load_chunk(q);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(&tslot)),
                 "r"(NCOL));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // input rows -> high and low parts of B = [Re | Im], zero past the tile's reduction end
  const int64_t ro = rowoff[g.t];
  if (tid < g.nch * 16) {
    const int l = tid;
    float2 v[S];
#pragma unroll
    for (int c = 0; c < S; ++c) v[c] = make_float2(0.f, 0.f);
    if (l < g.nk) {
      const int64_t R = ro + g.kbeg + l;
      const int local = g.kbeg + l;
      const float2* xs = (FWD || local >= g.k) ? Xsub + (int64_t)rows[R] * s : Wout + R * s;
#pragma unroll
      for (int c = 0; c < S; ++c)
        if (c < s) v[c] = xs[c];
      if (FWD) {
        const int2 cc = csrc[R];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int cr = h ? cc.y : cc.x;
          if (cr < 0) continue;
          const float2* w = Wout + (int64_t)cr * s;
#pragma unroll
          for (int c = 0; c < S; ++c)
            if (c < s) v[c] = make_float2(v[c].x + w[c].x, v[c].y + w[c].y);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < S; ++c) {
      const float reh = tc_hi(v[c].x), imh = tc_hi(v[c].y);
      const int o0 = tc_off(c, l, TC_SBO_B), o1 = tc_off(S + c, l, TC_SBO_B);
      *reinterpret_cast<float*>(sBh + o0) = reh;
      *reinterpret_cast<float*>(sBh + o1) = imh;
      *reinterpret_cast<float*>(sBl + o0) = tc_hi(v[c].x - reh);
      *reinterpret_cast<float*>(sBl + o1) = tc_hi(v[c].y - imh);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // B: generic writes, async-proxy reads
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t taddr = tslot;
  // kind::tf32: D f32, A and B tf32, both K-major, N = 2S, M = 128
  constexpr uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  const int per_plane = g.nr8 * 16;  // floats of one plane of a chunk
  for (int q = 0; q < g.nch; ++q) {
    const int r = q % TC_NRAW;
    bool okq = tc_wait(tc_smem(&full[r]), (q / TC_NRAW) & 1);
    if (okq && q >= 1) okq = tc_wait(tc_smem(&freeb), (q - 1) & 1);  // MMAs of chunk q - 1 done
    if (!okq) s_ok = 0;
    if (okq)
      for (int i = tid; i < 2 * per_plane; i += MF_TILE) {
        const int pl = i >= per_plane, e = i - pl * per_plane;
        const float x = *(reinterpret_cast<const float*>(raw + r * TC_STAGE + pl * TC_PLANE) + e);
        const float h = tc_hi(x);
        *(reinterpret_cast<float*>(wh + pl * TC_PLANE) + e) = h;
        *(reinterpret_cast<float*>(wl + pl * TC_PLANE) + e) = tc_hi(x - h);
      }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (!s_ok) break;
    if (tid == 0) {
      // every thread has read raw stage r: it takes the copy of chunk q + TC_NRAW
      if (q + TC_NRAW < g.nch) load_chunk(q + TC_NRAW);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t aReH = tc_smem(wh), aImH = aReH + TC_PLANE, aReL = tc_smem(wl), aImL = aReL + TC_PLANE;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const uint32_t kb = (uint32_t)(q * 4 + 2 * j) * 128;
        const uint64_t dReH = tc_desc(aReH + j * 256, 128, TC_SBO_A), dImH = tc_desc(aImH + j * 256, 128, TC_SBO_A);
        const uint64_t dReL = tc_desc(aReL + j * 256, 128, TC_SBO_A), dImL = tc_desc(aImL + j * 256, 128, TC_SBO_A);
        const uint64_t dbh = tc_desc(tc_smem(sBh) + kb, 128, TC_SBO_B), dbl = tc_desc(tc_smem(sBl) + kb, 128, TC_SBO_B);
        const uint32_t first = (q > 0 || j > 0) ? 1u : 0u;
        tc_mma(taddr, dReH, dbh, idesc, first);
        tc_mma(taddr, dReH, dbl, idesc, 1u);
        tc_mma(taddr, dReL, dbh, idesc, 1u);
        tc_mma(taddr + N, dImH, dbh, idesc, first);
        tc_mma(taddr + N, dImH, dbl, idesc, 1u);
        tc_mma(taddr + N, dImL, dbh, idesc, 1u);
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       tc_smem(&freeb))
                   : "memory");
    }
  }
  // `done` arrives once every MMA issued so far has completed
  if (tid == 0)
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem(&done))
                 : "memory");
  const bool fin = tc_wait(tc_smem(&done), 0);
  if (!fin) s_ok = 0;
  __syncthreads();
  const bool ok = s_ok != 0;
  if (!ok && tid == 0) {
    atomicExch(err, 1);
    // copies still in flight must land before the CTA's shared memory is released (bounded waits;
    // a stage whose chunk was already consumed passes at once)
    for (int q = max(0, issued - TC_NRAW); q < issued; ++q) tc_wait(tc_smem(&full[q % TC_NRAW]), (q / TC_NRAW) & 1);
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (ok) {
    const int m = tid;  // TMEM lane = output row of the tile
    const bool act = m < g.nr;
    const int rr = g.r0 + m;
    const int64_t Rg = ro + rr;
    const uint32_t lane_base = taddr + ((uint32_t)(warp * 32) << 16);
    uint32_t d1r[16], d1i[16], d2r[16], d2i[16];
#define HZ_TMEM_LD16(dst, col)                                                                                      \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];" \
               : "=r"(dst[0]), "=r"(dst[1]), "=r"(dst[2]), "=r"(dst[3]), "=r"(dst[4]), "=r"(dst[5]), "=r"(dst[6]),     \
                 "=r"(dst[7]), "=r"(dst[8]), "=r"(dst[9]), "=r"(dst[10]), "=r"(dst[11]), "=r"(dst[12]), "=r"(dst[13]), \
                 "=r"(dst[14]), "=r"(dst[15])                                                                       \
               : "r"(lane_base + (col)))
    HZ_TMEM_LD16(d1r, 0);
    HZ_TMEM_LD16(d1i, S);
    HZ_TMEM_LD16(d2r, N);
    HZ_TMEM_LD16(d2i, N + S);
#undef HZ_TMEM_LD16
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    if (act) {
#pragma unroll
      for (int c = 0; c < S; ++c) {
        if (c >= s) break;
        // Re(M b) = Re M Re b - Im M Im b,  Im(M b) = Re M Im b + Im M Re b
        float2 a = make_float2(__uint_as_float(d1r[c]) - __uint_as_float(d2i[c]),
                               __uint_as_float(d1i[c]) + __uint_as_float(d2r[c]));
        if (g.slot >= 0) {
          P[((int64_t)g.slot * MF_TILE + m) * s + c] = a;
        } else if (FWD) {
          if (rr < g.k) {
            Wout[Rg * s + c] = c_mul(a, Dinv[Doff[g.t] + rr]);
          } else {
            const int2 cc = csrc[Rg];
            if (cc.x >= 0) a = c_add(a, Wout[(int64_t)cc.x * s + c]);
            if (cc.y >= 0) a = c_add(a, Wout[(int64_t)cc.y * s + c]);
            Wout[Rg * s + c] = a;
          }
        } else {
          Xsub[(int64_t)rows[Rg] * s + c] = a;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(NCOL));
}

static inline unsigned blocks_for(int64_t work, int b) { return (unsigned)((work + b - 1) / b); }

template <bool FWD>
static void tc_launch(DevMF& mf, int l, float2* Xsub, int s, cudaStream_t st) {
  const int* ptr = FWD ? mf.ftc_ptr_h : mf.btc_ptr_h;
  const int tb = ptr[l], te = ptr[l + 1];
  if (te > tb) {
    k_mf_tile_tc<TS, FWD><<<te - tb, MF_TILE, tc_smem_bytes<TS>(), st>>>(
        (FWD ? mf.ftiles_tc : mf.btiles_tc) + tb, (FWD ? mf.ftc_off : mf.btc_off) + tb, mf.TC, mf.k, mf.f, mf.rowoff,
        mf.rows, mf.csrc, mf.Doff, (const float2*)mf.Dinv, Xsub, (float2*)mf.Wout, (float2*)mf.P, s, mf.tc_err);
    count_launch();
  }
}

// One level's SIMT tiles, and the sums of its split row blocks
template <bool FWD>
static void launch_tiles(DevMF& mf, int l, float2* Xsub, int s, cudaStream_t st) {
  const int* ptr = FWD ? mf.fs_ptr_h : mf.bs_ptr_h;
  const int nt = ptr[l + 1] - ptr[l];
  if (nt == 0) return;
  const bool half = (FWD ? mf.fhalf_h : mf.bhalf_h)[l] != 0 && nt >= MF_SHORT_LEVEL;
  const int rows = half ? MF_HALF : MF_TILE, tpr = half ? 2 : (nt < MF_SHORT_LEVEL ? 4 : 1);
  auto kern = half ? k_mf_tile<FWD, 2, MF_HALF> : (tpr == 4 ? k_mf_tile<FWD, 4, MF_TILE> : k_mf_tile<FWD, 1, MF_TILE>);
  launch_k(false, kern, (unsigned)nt, (unsigned)(rows * tpr), 0, st,
           (const int4*)((FWD ? mf.ftiles_s : mf.btiles_s) + ptr[l]), (const int*)mf.k, (const int*)mf.f,
           (const int64_t*)mf.rowoff, (const int64_t*)(FWD ? mf.Moff : mf.MToff),
           (const float2*)(FWD ? mf.M : mf.MT), (const int*)mf.rows, (const int2*)mf.csrc, (const int64_t*)mf.Doff,
           (const float2*)mf.Dinv, Xsub, (float2*)mf.Wout, (float2*)mf.P, s);
}
template <bool FWD>
static void launch_reduce(DevMF& mf, int l, float2* Xsub, int s, cudaStream_t st) {
  const int* ptr = FWD ? mf.frb_ptr_h : mf.brb_ptr_h;
  const int nrb = ptr[l + 1] - ptr[l];
  if (nrb == 0) return;
  launch_k(false, k_mf_reduce<FWD>, blocks_for((int64_t)nrb * MF_TILE * s, 256), 256, 0, st,
           (const int4*)((FWD ? mf.frb : mf.brb) + ptr[l]), nrb, (const int*)mf.k, (const int*)mf.f,
           (const int64_t*)mf.rowoff, (const int64_t*)mf.Doff, (const int*)mf.rows, (const int2*)mf.csrc,
           (const float2*)mf.Dinv, (float2*)mf.Wout, (const float2*)mf.P, Xsub, s);
}

// The tensor-core form of the sweeps: a level's SIMT tiles run on the side
// stream, concurrently with its tcgen05 tiles (they write disjoint outputs
// and partial slots); the level's reduce waits for both.
static void tile_solve(DevMF& mf, float2* Xsub, int s, cudaStream_t st) {
  auto level = [&](auto fwd, int l) {
    constexpr bool FWD = decltype(fwd)::value;
    cudaStream_t ss = mf.side ? mf.side : st;
    if (mf.side) {
      cudaEventRecord(mf.ev_fork, st);
      cudaStreamWaitEvent(mf.side, mf.ev_fork, 0);
    }
    launch_tiles<FWD>(mf, l, Xsub, s, ss);
    tc_launch<FWD>(mf, l, Xsub, s, st);
    if (mf.side) {
      cudaEventRecord(mf.ev_join, mf.side);
      cudaStreamWaitEvent(st, mf.ev_join, 0);
    }
    launch_reduce<FWD>(mf, l, Xsub, s, st);
  };
  for (int l = 0; l < mf.nlevels; ++l) level(std::true_type(), l);
  for (int l = mf.nlevels - 1; l >= 0; --l) level(std::false_type(), l);
}

// Opt the tensor-core kernels into their dynamic shared memory once, outside
// any stream capture (called from the factorisation).
static void tile_attrs() {
  const int tshm = (int)tc_smem_bytes<TS>();
  cudaFuncSetAttribute(k_mf_tile_tc<TS, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, tshm);
  cudaFuncSetAttribute(k_mf_tile_tc<TS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, tshm);
}

// Row length of the sub-vector and front vectors of a block of s columns. The
// tile form works on any width: padded to 16, blocks of 9 and 12 columns took
// 2.58 and 2.60 ms on the quarter workload against 2.16 and 2.25.
int sub_cols(const DevMF& mf, int s) { return mf_tc_usable(mf, s) ? s : sweep_cols(s); }

void mf_solve(DevMF& mf, void* Xsub, int s, cudaStream_t st) {
  if (mf_tc_usable(mf, s))
    tile_solve(mf, (float2*)Xsub, s, st);
  else
    sweep_solve(mf, Xsub, sweep_cols(s), st);
}

}  // namespace hz
