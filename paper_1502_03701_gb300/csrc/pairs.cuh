// FP32 pairs ("float-float", a value is hi + lo): conversions from and to
// double with integer operations only (no FP64-pipe work), exact FMA
// two-products (Dekker) and two-sum accumulation (Knuth), ~2^-48 relative.
#pragma once
#include <cuda_runtime.h>

struct ffn {
  float hi, lo;
};

// Exact split of a double into an FP32 pair with integer operations only
// (no FP64-pipe conversions): hi keeps the top 24 significant bits, lo the
// next bits rounded to 24 (|d - hi - lo| <= 2^-47 |d|).  Values below 2^-74
// keep hi only; values outside the FP32 range saturate.
__device__ __forceinline__ ffn ff_split(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7FF);
  const int ef = e - 1023 + 127;
  if (ef <= 0) return ffn{0.0f, 0.0f};
  if (ef >= 255) return ffn{__uint_as_float(sign | 0x7F800000u), 0.0f};
  const unsigned long long mant = b & 0xFFFFFFFFFFFFFull;
  const float hi = __uint_as_float(sign | ((unsigned)ef << 23) | (unsigned)(mant >> 29));
  float lo = 0.0f;
  const unsigned mlo = (unsigned)(mant & 0x1FFFFFFFu);
  if (mlo != 0u && e >= 949) {
    lo = __uint2float_rn(mlo) * __uint_as_float((unsigned)(e - 948) << 23);
    if (sign) lo = -lo;
  }
  return ffn{hi, lo};
}
// float -> double exactly, with integer operations
__device__ __forceinline__ double f2d_exact(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned ex = (u >> 23) & 0xFF;
  if (ex == 0) return 0.0;  // zero (FP32 denormals do not occur here)
  const unsigned long long b = ((unsigned long long)(u & 0x80000000u) << 32) |
                               ((unsigned long long)(ex - 127 + 1023) << 52) |
                               ((unsigned long long)(u & 0x7FFFFFu) << 29);
  return __longlong_as_double((long long)b);
}


// a + b for pairs (two-sum on the high parts, low parts added, renormalised)
__device__ __forceinline__ ffn ff_add(ffn a, ffn b) {
  float s = a.hi + b.hi;
  float bb = s - a.hi;
  float e = (a.hi - (s - bb)) + (b.hi - bb);
  e += a.lo + b.lo;
  float t = s + e;
  return ffn{t, e - (t - s)};
}
// acc += a * b: exact product of the high parts (FMA), cross terms in FP32,
// the high sum by two-sum; the low part collects all rounding errors
__device__ __forceinline__ void ff_acc_prod(ffn& acc, ffn a, ffn b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  const float s = acc.hi + p;
  const float bb = s - acc.hi;
  acc.lo += ((acc.hi - (s - bb)) + (p - bb)) + e;
  acc.hi = s;
}
__device__ __forceinline__ ffn ff_negate(ffn a) { return ffn{-a.hi, -a.lo}; }
__device__ __forceinline__ ffn ff_sub(ffn a, ffn b) { return ff_add(a, ff_negate(b)); }
// c * d as an unnormalised pair: the exact product of the high parts (FMA)
// plus the cross terms (the lo * lo term is below the pair's precision)
__device__ __forceinline__ ffn ff_prod(ffn c, ffn d) {
  const float p = c.hi * d.hi;
  float e = fmaf(c.hi, d.hi, -p);
  e = fmaf(c.hi, d.lo, fmaf(c.lo, d.hi, e));
  return ffn{p, e};
}
// d * 2^-sh split into a pair (exponents shifted with integer operations, so
// the scaling is exact); doubles whose scaled value falls below the double
// range give zero
__device__ __forceinline__ ffn ff_split_scaled(double d, int sh) {
  const long long b = __double_as_longlong(d);
  const int e = (int)((b >> 52) & 0x7FF);
  if (e == 0) return ffn{0.0f, 0.0f};
  const int es = e - sh;
  if (es <= 0) return ffn{0.0f, 0.0f};
  return ff_split(__longlong_as_double(b - ((long long)sh << 52)));
}
// float * 2^sh -> double exactly, with integer operations (zero below the
// double range)
__device__ __forceinline__ double f2d_exact_scaled(float f, int sh) {
  const unsigned u = __float_as_uint(f);
  const int ex = (int)((u >> 23) & 0xFF);
  if (ex == 0) return 0.0;
  const int E = ex - 127 + 1023 + sh;
  if (E <= 0) return 0.0;
  const unsigned long long b = ((unsigned long long)(u & 0x80000000u) << 32) | ((unsigned long long)E << 52) |
                               ((unsigned long long)(u & 0x7FFFFFu) << 29);
  return __longlong_as_double((long long)b);
}
__device__ __forceinline__ double ff_to_d_scaled(ffn a, int sh) {
  return f2d_exact_scaled(a.hi, sh) + f2d_exact_scaled(a.lo, sh);
}
__device__ __forceinline__ double ff_to_d(ffn a) { return f2d_exact(a.hi) + f2d_exact(a.lo); }
__device__ __forceinline__ ffn ff_warp_sum(ffn x) {
  for (int o = 16; o > 0; o >>= 1) {
    ffn y{__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o)};
    x = ff_add(x, y);
  }
  return x;
}

// ---------------------------------------------------------------------------
// Pair arithmetic of the derivative passes (rounding intrinsics, so that the
// compiler fuses nothing across the error terms).
// ---------------------------------------------------------------------------
// d to the nearest pair: hi is d rounded to 24 bits, lo the rest (29 bits,
// signed) rounded to 24, so |d - hi - lo| <= 2^-49 |d|.  Integer operations
// but one conversion: the FP64 pipe is not used.  |d| below 2^-126 gives zero,
// lo is kept from 2^-74 up; from 2^127 up and for NaN, hi is Inf or NaN.
__device__ __forceinline__ ffn ff2_split(double d) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
  const unsigned e = (h >> 20) & 0x7FFu;
  const unsigned long long t = (((unsigned long long)h << 32) | l) + 0x10000000ull;  // half a unit of hi
  const unsigned sign = h & 0x80000000u;
  // exponent rebased by 896 modulo 512: exact for results in [1, 254]
  unsigned hb = sign | (((unsigned)(t >> 29) - (384u << 23)) & 0x7FFFFFFFu);
  float lo = __int2float_rn((int)(l << 3) >> 3) * __uint_as_float(sign | ((unsigned)max((int)e - 948, 0) << 23));
  if (e - 897u >= 253u) {  // zero, tiny, huge, Inf or NaN
    hb = e < 897u ? sign : (sign | (e == 0x7FFu && ((h & 0xFFFFFu) | l) ? 0x7FC00000u : 0x7F800000u));
    lo = 0.0f;
  }
  return ffn{__uint_as_float(hb), lo};
}
__device__ __forceinline__ ffn ff2_norm(ffn a) {
  const float t = __fadd_rn(a.hi, a.lo);
  return ffn{t, __fsub_rn(a.lo, __fsub_rn(t, a.hi))};
}
__device__ __forceinline__ float ff2_two_sum(float a, float b, float& err) {
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}
// a + b; _u: low part not folded back into the high part
__device__ __forceinline__ ffn ff2_add_u(ffn a, ffn b) {
  float e;
  const float s = ff2_two_sum(a.hi, b.hi, e);
  return ffn{s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ ffn ff2_add(ffn a, ffn b) { return ff2_norm(ff2_add_u(a, b)); }
// w + c x: exact product of the high parts, cross terms, two-sum
__device__ __forceinline__ ffn ff2_fma_u(ffn c, ffn x, ffn w) {
  const float p = __fmul_rn(c.hi, x.hi);
  float e = __fmaf_rn(c.hi, x.hi, -p), t;
  e = __fmaf_rn(c.hi, x.lo, e);
  e = __fmaf_rn(c.lo, x.hi, e);
  const float s = ff2_two_sum(w.hi, p, t);
  return ffn{s, __fadd_rn(__fadd_rn(t, w.lo), e)};
}
__device__ __forceinline__ ffn ff2_fma(ffn c, ffn x, ffn w) { return ff2_norm(ff2_fma_u(c, x, w)); }
// hi + lo in FP64 with integer conversions and one add; Inf and NaN are kept
__device__ __forceinline__ double ff2_to_d(ffn a) {
  const unsigned u = __float_as_uint(a.hi);
  const double d = f2d_exact(a.hi) + f2d_exact(a.lo);
  if ((u & 0x7F800000u) != 0x7F800000u) return d;
  return __hiloint2double((int)((u & 0x80000000u) | 0x7FF00000u | ((u & 0x7FFFFFu) ? 0x80000u : 0u)), 0);
}
