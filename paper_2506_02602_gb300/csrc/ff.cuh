// ff.cuh -- double-float arithmetic: a value held as the unevaluated sum of two fp32
// numbers (about 48 significant bits), on the FP32 pipe.
//
// On GB300 a warp's FP64 instruction occupies its sub-partition's FP64 lanes for 64
// cycles (measured, whatever the instruction-level parallelism); an FP32 add or FMA takes
// one.  The error-free transformations below (Knuth's two-sum, Dekker's fast two-sum, the
// FMA two-product; T. J. Dekker, Numer. Math. 18 (1971) 224-242) make a double-float
// multiply-add about 12 FP32 instructions, a fifth of the FP64 pipe's time for one DFMA.
// Every step is written with rounding intrinsics, so no multiply-add is contracted and
// every kernel computes the same bits.
#pragma once

#include <cstdint>

#include "fastmath.cuh"

namespace chem {

// Per-block copy of k_ln_ff for ff_log, filled by load_ln_ff (all threads, then a barrier).
__shared__ float4 s_ln_ff[65];
__device__ __forceinline__ void load_ln_ff() {
  for (int i = threadIdx.x; i < 65; i += blockDim.x)
    s_ln_ff[i] = make_float4(k_ln_ff[i][0], k_ln_ff[i][1], k_ln_ff[i][2], 0.0f);
}

struct ff {
  float h, l;
};

__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }

// a + b exactly, any magnitudes (6 operations)
__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = fadd(a, b), t = fsub(s, a);
  return {s, fadd(fsub(a, fsub(s, t)), fsub(b, t))};
}
// a + b exactly for |a| >= |b| (3 operations)
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
  const float s = fadd(a, b);
  return {s, fsub(b, fsub(s, a))};
}

// products: relative error about 2^-46 of |a b|; the result's low part may exceed half an
// ulp of its high part by a few ulps (callers renormalise where that matters)
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = fmul(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  return {p, __fmaf_rn(a.l, b.h, e)};
}
__device__ __forceinline__ ff ff_norm(ff a) { return fast_two_sum(a.h, a.l); }
// a + b without renormalisation (the low parts just accumulate)
__device__ __forceinline__ ff ff_acc(ff a, ff b) {
  const ff s = two_sum(a.h, b.h);
  return {s.h, fadd(a.l, fadd(s.l, b.l))};
}

// Two double-floats side by side on the packed FP32 instructions (f32x2: two operations per
// issued instruction at the FP32 pipe's full rate): {h.x, l.x} and {h.y, l.y}.
struct ff2 {
  float2 h, l;
};
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ ff2 both(ff a) { return {both(a.h), both(a.l)}; }
__device__ __forceinline__ ff2 two_sum(float2 a, float2 b) {
  const float2 s = add2(a, b), t = sub2(s, a);
  return {s, add2(sub2(a, sub2(s, t)), sub2(b, t))};
}
__device__ __forceinline__ ff2 ff_norm(ff2 a) {
  const float2 s = add2(a.h, a.l);
  return {s, sub2(a.l, sub2(s, a.h))};
}
__device__ __forceinline__ ff2 ff_acc(ff2 a, ff2 b) {
  const ff2 s = two_sum(a.h, b.h);
  return {s.h, add2(a.l, add2(s.l, b.l))};
}
__device__ __forceinline__ ff2 ff_mul(ff2 a, float2 b) {
  const float2 p = __fmul2_rn(a.h, b);
  return {p, __ffma2_rn(a.l, b, __ffma2_rn(a.h, b, make_float2(-p.x, -p.y)))};
}
__device__ __forceinline__ ff2 ff_mul(ff2 a, ff2 b) {
  const float2 p = __fmul2_rn(a.h, b.h);
  float2 e = __ffma2_rn(a.h, b.h, make_float2(-p.x, -p.y));
  e = __ffma2_rn(a.h, b.l, e);
  return {p, __ffma2_rn(a.l, b.h, e)};
}

// An fp64 value as a pair: h the value truncated to 24 bits, l the remaining 29 bits
// rounded to 24, on the integer pipe (no FP64 instruction).  Magnitudes below 2^-126 go
// to zero, as in d2f; infinities and NaNs stay in h.
__device__ __forceinline__ ff d2ff(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t a = hi & 0x7fffffffu, sign = hi & 0x80000000u;
  uint32_t r = ((a - 0x38000000u) << 3) | (lo >> 29);
  const int es = (int)(a >> 20) - 948;  // exponent field of 2^(e - 52) in fp32
  float l = fmul((float)(int)(lo & 0x1fffffffu), __uint_as_float((uint32_t)es << 23));
  const bool over = a >= 0x47f00000u, tiny = a < 0x38100000u;
  if (over) r = (a > 0x7ff00000u || (a == 0x7ff00000u && lo != 0u)) ? 0x7fc00000u : 0x7f800000u;
  if (tiny) r = 0u;
  if (over || es <= 0) l = 0.0f;
  return {__uint_as_float(r | sign), __uint_as_float(__float_as_uint(l) ^ sign)};
}
__device__ __forceinline__ double ff2d(ff a) { return __dadd_rn(f2d(a.h), f2d(a.l)); }

// ln x of a positive normal pair, absolute error below 8.5e-14 (rms 8e-15) at |ln x| < 16: x = 2^e f,
// c_j = 1 / (1 + j/64) in fp32 for the nearest 64th of the fraction, r = f c_j - 1
// (|r| <= 1/128; the product's rounding error is kept) and ln(1 + r) with r - r^2/2 in
// double-float and the terms from r^3 on in fp32; -ln c_j from a table of pairs in shared
// memory (s_ln_ff).
__device__ __forceinline__ ff ff_log(ff x) {
  const uint32_t b = __float_as_uint(x.h);
  const int e = (int)(b >> 23) - 127;
  const float fh = __uint_as_float((b & 0x007fffffu) | 0x3f800000u);
  const float fl = fmul(x.l, __uint_as_float((uint32_t)(127 - e) << 23));
  const int j = (int)(((b & 0x007fffffu) + 0x00010000u) >> 17);
  const float4 t = s_ln_ff[j];
  const float p = fmul(fh, t.x);
  const ff r = fast_two_sum(fsub(p, 1.0f), __fmaf_rn(fl, t.x, __fmaf_rn(fh, t.x, -p)));
  const float s = fmul(r.h, r.h), se = __fmaf_rn(r.h, r.h, -s);
  float q = __fmaf_rn(r.h, -1.0f / 6.0f, 0.2f);
  q = __fmaf_rn(r.h, q, -0.25f);
  q = __fmaf_rn(r.h, q, 1.0f / 3.0f);
  // r^3 (1/3 - r/4 + ...) and the low parts of r - r^2/2
  float lo = __fmaf_rn(fmul(s, r.h), q, fsub(r.l, __fmaf_rn(r.h, r.l, fmul(0.5f, se))));
  // e ln2 = e kLn2A (exact: 16 bits) + e kLn2B (with its rounding error) + e kLn2C
  const float ef = (float)e, eb = fmul(ef, kLn2B);
  lo = fadd(lo, __fmaf_rn(ef, kLn2C, __fmaf_rn(ef, kLn2B, -eb)));
  // the small terms first: their low parts are then small too
  const ff a = two_sum(fmul(ef, kLn2A), t.y);
  const ff c = fast_two_sum(r.h, fmul(-0.5f, s));
  const ff d = two_sum(c.h, eb);
  const ff g = two_sum(a.h, d.h);
  return fast_two_sum(g.h, fadd(fadd(a.l, g.l), fadd(fadd(c.l, d.l), fadd(lo, t.z))));
}

}  // namespace chem
