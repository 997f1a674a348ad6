// Double-float device helpers (pairs of FP32 numbers standing for one FP64
// value; see df.cu for the scheme and its error bounds), shared by the
// double-float product (df.cu) and the double-float Arnoldi process
// (krylov.cu).
#pragma once
#include <cuda_runtime.h>

#include "f32x2.cuh"

namespace hz {

// Conversions between FP64 and double-float by the IEEE-754 bit layouts, so
// that they issue integer instructions instead of FP64-pipe conversions.
//
// x -> (hi, lo): hi keeps the sign, exponent and leading 24 significant bits
// of x (truncated); lo is the remaining 29 bits rounded to 23, built from its
// bits as (1 + r) 2^(E-23) - 2^(E-23) (one exact FP32 subtraction), so that
// |hi + lo - x| <= 2^-47 |x|. Zeros and FP64 subnormals give (0, 0); values
// outside [2^-103, 2^128) fall back to one rounding (lo = 0).
static __device__ __forceinline__ float2 df_split(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7FF);
  if (e == 0) return make_float2(__uint_as_float(sign), 0.f);
  const int fe = e - 1023 + 127;
  if (fe <= 23 || fe >= 255) return make_float2(__double2float_rn(x), 0.f);
  const unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  const float hi = __uint_as_float(sign | ((unsigned)fe << 23) | (unsigned)(m >> 29));
  const unsigned base = (unsigned)(fe - 23) << 23;                        // 2^(E-23) as FP32 bits
  const unsigned r23 = (unsigned)(((m & 0x1FFFFFFFull) + 32ull) >> 6);      // rounded, may carry to 2^23
  const float lo = __fsub_rn(__uint_as_float(base + r23), __uint_as_float(base));
  return make_float2(hi, sign ? -lo : lo);
}

// FP32 -> FP64 (exact)
static __device__ __forceinline__ double f2d(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xFFu;
  const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
  if ((u & 0x7FFFFFFFu) == 0) return __longlong_as_double((long long)sign);
  if (e == 0 || e == 255) return (double)f;  // subnormal, inf, nan
  return __longlong_as_double(
      (long long)(sign | ((unsigned long long)(e - 127 + 1023) << 52) | ((unsigned long long)(u & 0x7FFFFFu) << 29)));
}

// hi + lo as FP64 for a renormalised pair (|lo| <= ulp(hi)), by integer
// instructions: hi's significand moved up by 29 bits plus lo in units of its
// last place, rounded to nearest: the same bits as the FP64 sum. Pairs whose
// sum falls below hi's power of two, others, and values outside the range in
// which the units are normal FP32 numbers, go through the FP64 pipe.
static __device__ __forceinline__ double df_join(float hi, float lo) {
  const unsigned u = __float_as_uint(hi);
  const int e = (int)((u >> 23) & 0xFFu);  // hi = 1.f 2^(e - 127)
  if (e < 60 || e > 190 || fabsf(lo) > __uint_as_float((unsigned)(e - 23) << 23)) return f2d(hi) + f2d(lo);
  // one unit = 2^(e - 127 - 52); lo in units, |lo| <= 2^29
  const int l = __float2int_rn(__fmul_rn(lo, __uint_as_float((unsigned)(306 - e) << 23)));
  long long m = ((long long)((u & 0x7FFFFFu) | 0x800000u)) << 29;
  m += (u >> 31) ? -(long long)l : (long long)l;
  long long ex = e - 127 + 1023;
  if (m < (1ll << 52)) return f2d(hi) + f2d(lo);  // one more bit would be needed
  if (m >= (1ll << 53)) {                         // the next power of two itself
    m >>= 1;
    ++ex;
  }
  return __longlong_as_double((long long)((unsigned long long)(u & 0x80000000u) << 32) | (ex << 52) |
                              (m & 0xFFFFFFFFFFFFFll));
}

// (sh, sl) += (ah + al) (xh + xl); the al*xl term (2^-48 relative) is dropped
static __device__ __forceinline__ void df_mac(float& sh, float& sl, float ah, float al, float xh, float xl) {
  const float p = __fmul_rn(ah, xh);
  float e = __fmaf_rn(ah, xh, -p);  // exact: ah*xh = p + e
  e = __fmaf_rn(ah, xl, e);
  e = __fmaf_rn(al, xh, e);
  const float t = __fadd_rn(sh, p);  // TwoSum: sh + p = t + err exactly
  const float z = __fsub_rn(t, sh);
  const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, z)), __fsub_rn(p, z));
  sl = __fadd_rn(sl, __fadd_rn(err, e));
  sh = t;
}

// The same on both halves of packed pairs, bit for bit; na = -ah. (The
// subtractions take p negated: s + p = s - np.)
static __device__ __forceinline__ void df_add2(pair2& sh, pair2& sl, pair2 np, pair2 e) {
  const pair2 t = sub2(sh, np);
  const pair2 z = sub2(t, sh);
  const pair2 nerr = sub2(add2(np, z), sub2(sh, sub2(t, z)));  // -((sh - (t - z)) + (p - z))
  sl = add2(sl, sub2(e, nerr));
  sh = t;
}
static __device__ __forceinline__ void df_mac2(pair2& sh, pair2& sl, pair2 ah, pair2 na, pair2 al, pair2 xh, pair2 xl) {
  const pair2 np = mul2(na, xh);
  df_add2(sh, sl, np, fma2(al, xh, fma2(ah, xl, fma2(ah, xh, np))));
}
// xl = 0
static __device__ __forceinline__ void df_mac2(pair2& sh, pair2& sl, pair2 ah, pair2 na, pair2 al, pair2 xh) {
  const pair2 np = mul2(na, xh);
  df_add2(sh, sl, np, fma2(al, xh, fma2(ah, xh, np)));
}

// renormalise (h, l) so that |l| is at most half an ulp of h (Fast2Sum; |h| >= |l| or h = 0)
static __device__ __forceinline__ void df_norm(float& h, float& l) {
  const float t = __fadd_rn(h, l);
  l = __fsub_rn(l, __fsub_rn(t, h));
  h = t;
}

// (h, l) = (ah + al) (bh + bl), renormalised; the al*bl term is dropped
static __device__ __forceinline__ void df_mul(float& h, float& l, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  h = p;
  l = e;
  df_norm(h, l);
}

}  // namespace hz
