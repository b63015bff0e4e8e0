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
// d to the nearest pair: hi is d rounded to 24 bits (half away from zero), lo
// the rest (29 bits, signed) rounded to 24, so |d - hi - lo| <= 2^-49 |d|.
// Integer operations but one conversion: the FP64 pipe is not used.  |d| below
// 2^-126 gives zero (to 2^-146), lo is kept from 2^-74 up; from 2^127 up and
// for Inf and NaN, hi is Inf or NaN.  up: d 2^u is split instead, exactly, with
// up = u << 20 and |u| <= kPairMaxUp; the limits hold for that product.
constexpr int kPairMaxUp = 400;
__device__ __forceinline__ ffn ff2_split(double d, int up = 0) {
  const unsigned h = (unsigned)__double2hiint(d), l = (unsigned)__double2loint(d);
  const unsigned a = h & 0x7FFFFFFFu, tl = l + 0x10000000u;  // plus half a unit of hi
  // exponent rebased by 896, clamped to the FP32 range
  const int th = min(max((int)(a + (tl < l ? 1u : 0u)) - ((896 << 20) - up), 0), 255 << 20);
  const float hi = __uint_as_float(__funnelshift_l(tl, (unsigned)th, 3) | (h & 0x80000000u));
  // the low 29 bits as a signed integer, in units of 2^(e - 52)
  const unsigned sc = ((unsigned)max((int)a - ((948 << 20) - up), 0) << 3) & 0x7F800000u;
  return ffn{hi, __fmul_rn(__int2float_rn((int)(l << 3) >> 3), __uint_as_float(sc | (h & 0x80000000u)))};
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
// hi + lo in FP64 (normalised pair), correctly rounded to 53 bits but for one
// unit, with integer operations: lo is rounded to units of hi's 52-bit
// mantissa and added to hi's bit pattern.  A power of two with lo of the other
// sign (the unit halves below it) takes an FP64 add; Inf and NaN are kept.
__device__ __forceinline__ double ff2_to_d(ffn a) {
  const unsigned u = __float_as_uint(a.hi), ex = (u >> 23) & 0xFFu, m = u & 0x7FFFFFu;
  if (ex <= 52u || ex >= 200u || m == 0u) {  // tiny, huge, zero, Inf, NaN or a power of two
    if (ex != 0xFFu) return f2d_exact(a.hi) + f2d_exact(a.lo);
    return __hiloint2double((int)((u & 0x80000000u) | 0x7FF00000u | (m ? 0x80000u : 0u)), 0);
  }
  // lo / 2^(e - 52) with hi's sign taken off; |.| <= 2^28
  const float sc = __uint_as_float((u & 0x80000000u) | ((306u - ex) << 23));
  const int li = __float2int_rn(__fmul_rn(a.lo, sc));
  const unsigned long long b = ((unsigned long long)((u & 0x80000000u) | ((ex + 896u) << 20) | (m >> 3)) << 32) |
                               (unsigned long long)(m << 29);
  return __longlong_as_double((long long)(b + (unsigned long long)(long long)li));
}

// ---------------------------------------------------------------------------
// Two pairs side by side (the real and imaginary components), on the packed
// FP32 instructions of sm_100: one issue slot for two operations.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 v2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 v2_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 v2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 v2_sub(float2 a, float2 b) { return __fadd2_rn(a, v2_neg(b)); }
__device__ __forceinline__ float2 v2_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 v2_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float v2_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
struct ffn2 {
  float2 hi, lo;
};
__device__ __forceinline__ ffn2 ff2_dup(ffn a) { return ffn2{v2(a.hi), v2(a.lo)}; }
__device__ __forceinline__ ffn2 ff2_zero2() { return ffn2{v2(0.0f), v2(0.0f)}; }
__device__ __forceinline__ ffn2 ff2_neg(ffn2 a) { return ffn2{v2_neg(a.hi), v2_neg(a.lo)}; }
// in 16 (8) bytes, highs first; a slot of the derivative scratch holds (re.hi, re.lo, im.hi, im.lo)
__device__ __forceinline__ float4 ff2_pack(ffn2 a) { return make_float4(a.hi.x, a.hi.y, a.lo.x, a.lo.y); }
__device__ __forceinline__ ffn2 ff2_unpack(float4 a) { return ffn2{make_float2(a.x, a.y), make_float2(a.z, a.w)}; }
__device__ __forceinline__ float4 ff2_to_slot(ffn2 a) { return make_float4(a.hi.x, a.lo.x, a.hi.y, a.lo.y); }
__device__ __forceinline__ ffn2 ff2_from_slot(float4 a) { return ffn2{make_float2(a.x, a.z), make_float2(a.y, a.w)}; }
__device__ __forceinline__ float2 ff2_pack(ffn a) { return make_float2(a.hi, a.lo); }
__device__ __forceinline__ ffn ff2_unpack(float2 a) { return ffn{a.x, a.y}; }
__device__ __forceinline__ float2 ff2_to_slot(ffn a) { return make_float2(a.hi, a.lo); }
__device__ __forceinline__ ffn ff2_from_slot(float2 a) { return ffn{a.x, a.y}; }
__device__ __forceinline__ ffn ff2_neg(ffn a) { return ffn{-a.hi, -a.lo}; }
__device__ __forceinline__ ffn2 ff2_split(double2 d, int up = 0) {
  const ffn a = ff2_split(d.x, up), b = ff2_split(d.y, up);
  return ffn2{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)};
}
__device__ __forceinline__ double2 ff2_to_d(ffn2 a) {
  return make_double2(ff2_to_d(ffn{a.hi.x, a.lo.x}), ff2_to_d(ffn{a.hi.y, a.lo.y}));
}
__device__ __forceinline__ ffn2 ff2_norm(ffn2 a) {
  const float2 t = v2_add(a.hi, a.lo);
  return ffn2{t, v2_sub(a.lo, v2_sub(t, a.hi))};
}
__device__ __forceinline__ float2 ff2_two_sum(float2 a, float2 b, float2& err) {
  const float2 s = v2_add(a, b), bb = v2_sub(s, a);
  err = v2_add(v2_sub(a, v2_sub(s, bb)), v2_sub(b, bb));
  return s;
}
__device__ __forceinline__ ffn2 ff2_add_u(ffn2 a, ffn2 b) {
  float2 e;
  const float2 s = ff2_two_sum(a.hi, b.hi, e);
  return ffn2{s, v2_add(e, v2_add(a.lo, b.lo))};
}
__device__ __forceinline__ ffn2 ff2_add(ffn2 a, ffn2 b) { return ff2_norm(ff2_add_u(a, b)); }
__device__ __forceinline__ ffn2 ff2_fma_u(ffn2 c, ffn2 x, ffn2 w) {
  const float2 p = v2_mul(c.hi, x.hi);
  float2 e = v2_fma(c.hi, x.hi, v2_neg(p)), t;
  e = v2_fma(c.hi, x.lo, e);
  e = v2_fma(c.lo, x.hi, e);
  const float2 s = ff2_two_sum(w.hi, p, t);
  return ffn2{s, v2_add(v2_add(t, w.lo), e)};
}
__device__ __forceinline__ ffn2 ff2_fma(ffn2 c, ffn2 x, ffn2 w) { return ff2_norm(ff2_fma_u(c, x, w)); }
