// fastmath.cuh -- fp64 device math for the FP64-pipe-bound kernels: table-driven exp
// and log, Newton-Raphson reciprocals, and fp32 <-> fp64 conversions, compares and
// clamps on the integer pipe.
//
// On GB300 the FP64 pipe issues 2 lanes per clock per SM, and a library fp64 exp takes
// about 20 of those slots (log about 37).  The right-hand side's ~50 exponentials, its logarithms
// and its sums of products run in 64-bit fixed point on the integer pipe (exp2_q52, log2_q58,
// DotQ).  Arguments outside the fixed-point forms' ranges take exp_t and log_t, which
// follow Tang's table-driven methods (ACM TOMS 15 (1989) 144-157 for exp, 16 (1990)
// 378-400 for log) with Taylor polynomials, in about 10 FP64 operations each; the
// exponent and table-index arithmetic runs on the integer pipe and the 128-entry (exp)
// and 65-entry (log) tables live in shared memory.  Accuracy is about 1 ulp on the
// ranges used (checked against the CUDA library functions by the GPU tests through
// chem_diag_math).
#pragma once

#include <cstdint>

#include "math_tables.cuh"

namespace chem {

// Per-block copies of the tables: divergent table reads from shared memory cost far
// less latency than L1 round trips.  Every kernel that calls exp_t / log_t fills them
// first with load_math_tables() (all threads, then a barrier).
__shared__ double s_exp2_128[128];
__shared__ double s_log_inv[65];
__shared__ double s_log_tab[65];
__shared__ double s_log_tab_m1[65];

__device__ __forceinline__ void load_math_tables() {
  for (int i = threadIdx.x; i < 128; i += blockDim.x) {
    s_exp2_128[i] = k_exp2_128[i];
    if (i < 65) {
      s_log_inv[i] = k_log_inv[i];
      s_log_tab[i] = k_log_tab[i];
      s_log_tab_m1[i] = k_log_tab_m1[i];
    }
  }
  __syncthreads();
}

// x is a NaN, on the integer pipe
__device__ __forceinline__ bool is_nan(double x) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}

// x clamped to [-lim, lim] for lim > 0 (a NaN gives +-lim)
__device__ __forceinline__ double clamp_abs(double x, double lim) {
  const long long b = __double_as_longlong(x);
  const long long l = __double_as_longlong(lim);
  return (b & 0x7fffffffffffffffLL) > l ? __longlong_as_double((b & (long long)0x8000000000000000ULL) | l) : x;
}

// ---- exponentials in fixed point, on the integer pipe ----
// A 64-bit number in units of 2^-52 (Q52) stands for a base-2 logarithm.  Its first two tens of
// fraction bits index tables (8 KB each in shared memory) of 2^(j/2^10) and 2^(k/2^20) - 1, and
// the last 32, r < 2^-20, give 2^r - 1 as v + v^2/2 with v = r ln2.  No FP64 instruction, two wide
// and five high multiplies, and at most 0.51 ulp off: 32 instructions.
// (With one table and r < 2^-10 the terms to r^4, half of them in fp32, and their alignment took
// about twice as many.)

// Per-block copies of k_exp2_hi and k_exp2_lo, filled by load_exp2_tables().
__shared__ unsigned long long s_exp2_hi[1024], s_exp2_lo[1024];

__device__ __forceinline__ void load_exp2_tables() {
  for (int i = threadIdx.x; i < 1024; i += blockDim.x) {
    s_exp2_hi[i] = k_exp2_hi[i];
    s_exp2_lo[i] = k_exp2_lo[i];
  }
  __syncthreads();
}

__device__ __forceinline__ unsigned long long mul_wide(uint32_t a, uint32_t b) { return (unsigned long long)a * b; }

// 2^(y 2^-52 + yx 2^-84) for |y| < 1021 2^52; yx = 0 unless kLong
template <bool kLong = false>
__device__ __forceinline__ double exp2_q52_body(long long y, uint32_t yx = 0) {
  const uint32_t yl = (uint32_t)y, yh = (uint32_t)(y >> 32);
  const unsigned long long t = s_exp2_hi[(yh >> 10) & 1023], s0 = s_exp2_lo[yh & 1023];
  unsigned long long v = mul_wide(yl, kLn2Q64Hi) + __umulhi(yl, kLn2Q64Lo);  // units of 2^-84
  if constexpr (kLong) v += __umulhi(yx, kLn2Q64Hi);
  const uint32_t vh = (uint32_t)(v >> 32);
  const unsigned long long w = v + mul_wide(__umulhi(vh, vh), 2048u);  // + v^2/2
  // (1 + s0) (1 + w) - 1 in units of 2^-64
  const unsigned long long s = s0 + (w >> 20) + mul_wide(__umulhi((uint32_t)(s0 >> 22), (uint32_t)(w >> 32)), 4u);
  const uint32_t th = (uint32_t)(t >> 32), tl = (uint32_t)t, sh = (uint32_t)(s >> 32), sl = (uint32_t)s;
  const unsigned long long u = t + mul_wide(th, sh) + __umulhi(th, sl) + __umulhi(tl, sh);
  unsigned long long p = u >> 11;  // 53 bits, rounded
  if constexpr (kLong) p |= (unsigned long long)(u < t) << 53;  // less than half an ulp below the next power of 2
  // the leading bit, or a carry, adds to the exponent
  return __hiloint2double((int)((uint32_t)(p >> 32) + (yh & 0xfff00000u) + (1022u << 20)), (int)(uint32_t)p);
}

// Out of line, as exp_t: one copy of the code; two at a time where there are two, whose chains
// of dependent instructions then overlap.
static __device__ __noinline__ double exp2_q52(long long y) { return exp2_q52_body(y); }
static __device__ __noinline__ double2 exp2_q52(long long y0, long long y1) {
  return make_double2(exp2_q52_body(y0), exp2_q52_body(y1));
}

// exp(x) for the general form of the right-hand side.  |x| < 700: x log2(e) in units of 2^-84 from a
// 128-bit product and the exponential above, 0.51 ulp, without FP64 instructions.  Beyond, Tang's
// method, about 1 ulp: x = (128 m + j) ln2/128 + r, |r| <= ln2/256,
// e^r - 1 by its degree-5 Taylor polynomial (truncation below 6e-19 relative), and the
// scale 2^m added to the exponent field of the table entry 2^(j/128) on the integer
// pipe (10 FP64-pipe operations in all).  Arguments beyond +-710 are first clamped there
// on the integer pipe, so they still give +inf above and a positive value below 1e-307
// below, however large; a NaN stays NaN.  Kept out of line, one copy for its many calls.
static __device__ __noinline__ double exp_t(double x) {
  const uint32_t ah = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  if (ah < 0x4085e000u) {  // |x| < 700
    const unsigned long long m =
        (((unsigned long long)__double_as_longlong(x) & 0x000fffffffffffffull) | 0x0010000000000000ull) << 11;
    const int n = 1033 - (int)(ah >> 20);  // m = |x| 2^(53 + n), n >= 1
    const unsigned long long p = m * kLog2E_q127Hi, lo = p + __umul64hi(m, kLog2E_q127Lo);
    const unsigned long long hi = __umul64hi(m, kLog2E_q127Hi) + (lo < p);
    long long y = n < 64 ? (long long)(hi >> n) : 0;
    uint32_t yx = n < 64 ? (uint32_t)(((hi << (64 - n)) | (lo >> n)) >> 32) : (uint32_t)(hi >> min(n - 32, 63));
    if (__double2hiint(x) < 0) {
      y = -y - (yx != 0u);
      yx = 0u - yx;
    }
    return exp2_q52_body<true>(y, yx);
  }
  const long long kLim = 0x40863000'00000000LL;  // 710.0
  const long long b = __double_as_longlong(x);
  const long long ab = b & 0x7fffffffffffffffLL;
  if (ab > kLim && ab <= 0x7ff0000000000000LL) x = __longlong_as_double((b & (long long)0x8000000000000000ULL) | kLim);
  const double kShift = 6755399441055744.0;  // 1.5 * 2^52: rounds to an integer in the low bits
  const double t = fma(x, kInvLn2x128, kShift);
  const int k = min(max(__double2loint(t), -130816), 130943);  // 2^(k>>7) stays a normal double
  const double kd = (double)k;
  double r = fma(-kd, kLn2d128Hi, x);
  r = fma(-kd, kLn2d128Lo, r);
  // e^r - 1 = r + r^2/2 + r^3/6 + r^4/24 + r^5/120
  double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  p = fma(r, p, 1.0 / 6.0);
  p = fma(r, p, 0.5);
  p = fma(r, p, 1.0);
  p = r * p;
  const double tj = s_exp2_128[k & 127];
  const double ts = __hiloint2double(__double2hiint(tj) + ((k >> 7) << 20), __double2loint(tj));
  return fma(ts, p, ts);
}

// |x| in units of 2^-Q, truncated, for |x| < 2^(62 - Q + 1).
template <int Q>
__device__ __forceinline__ unsigned long long abs_q(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  const unsigned long long m = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 10;
  return m >> min(62 - Q - e, 63);
}

// x in Q52, limited to +-1009.9 (a factor e^+-700); a NaN gives a limit, so callers look for it
__device__ __forceinline__ long long to_q52(double x) {
  const long long v = (long long)abs_q<52>(clamp_abs(x, 1009.875));
  return __double2hiint(x) < 0 ? -v : v;
}

// x in units of 2^-Q kept within +-1020 by its upper word
template <int Q>
__device__ __forceinline__ long long limit_q(long long x) {
  const int lim = 1019 << (Q - 32), h = min(max((int)(x >> 32), -lim), lim);
  return (long long)(((unsigned long long)(uint32_t)h << 32) | (uint32_t)x);
}

// ---- sums of products in fixed point ----
// A 64-bit number is split into its upper 32 bits (signed) and the top 32 - D of its lower 32
// bits; of the product of two such numbers the upper x upper part and the two cross parts
// accumulate in 64 bits, one IMAD.WIDE each and nothing else: 15 cycles of a sub-partition a
// term on GB300 against 64 for an FP64 multiply-add.  What is dropped is below 2^(2 D - 64) of
// a unit of the result; callers bound their operands so that neither sum overflows.
template <int D>
struct Limbs { int h, l; };

template <int D>
__device__ __forceinline__ Limbs<D> limbs(long long v) { return {(int)(v >> 32), (int)((uint32_t)v >> D)}; }

// The same with the lower half in [-2^31, 2^31) and its limb signed, so that what is dropped has no
// bias.  v + 2^31 must not overflow.
template <int D>
__device__ __forceinline__ Limbs<D> limbs_centred(long long v) {
  return {(int)((unsigned long long)v >> 32) + (int)((uint32_t)v >> 31), (int)(uint32_t)v >> D};
}

template <int D>
struct DotQ {
  long long h, x;
  __device__ __forceinline__ void add(int ch, int cl, const Limbs<D> &p) {
    h += (long long)ch * p.h;
    x += (long long)ch * p.l;
    x += (long long)cl * p.h;
  }
  __device__ __forceinline__ long long value() const { return h + (x >> (32 - D)); }  // sum / 2^64
  // the same modulo 2^64 with F more bits
  template <int F>
  __device__ __forceinline__ unsigned long long fine() const {
    return ((unsigned long long)h << F) + (unsigned long long)(x >> (32 - D - F));
  }
};

// m t 2^-63 for 0 <= t < 2^63
__device__ __forceinline__ long long mul_q63(long long m, long long t) {
  const int mh = (int)(m >> 32), ml = (int)((uint32_t)m >> 1), th = (int)(t >> 32), tl = (int)((uint32_t)t >> 1);
  return (((long long)mh * th) << 1) + (((long long)mh * tl + (long long)ml * th) >> 30);
}

// The same from centred limbs, rounded; fine() is modulo 2^64, with F more bits.
struct MulQ {
  long long h, x;
  __device__ __forceinline__ MulQ(long long m, const Limbs<1> &t) {
    const Limbs<1> a = limbs_centred<1>(m);
    h = (long long)a.h * t.h;
    x = (long long)a.h * t.l + (1ll << 29);
    x += (long long)a.l * t.h;
  }
  __device__ __forceinline__ long long value() const { return (h << 1) + (x >> 30); }
  template <int F>
  __device__ __forceinline__ unsigned long long fine() const {
    return ((unsigned long long)h << (1 + F)) + (unsigned long long)((x - (1ll << 29)) >> (30 - F));
  }
};

// Per-block copies of k_log2_c and k_log2_q58, filled by load_log2_table().
__shared__ unsigned short s_log2_c[256];
__shared__ long long s_log2_q58[256];

__device__ __forceinline__ void load_log2_table() {
  for (int i = threadIdx.x; i < 256; i += blockDim.x) {
    s_log2_c[i] = k_log2_c[i];
    s_log2_q58[i] = k_log2_q58[i];
  }
  __syncthreads();
}

// log2 x = e + f, f in units of 2^-58, for positive normal x, at most 6 units off: x = 2^e (1 + ..),
// r = x 2^-e c_j - 1 exact in units of 2^-71 (|r| < 2^-8.9), log2(1 + r) with the terms from r^4
// on in fp32.
__device__ __forceinline__ long long log2_parts(double x, int &e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  e = (int)(b >> 52) - 1023;
  const int j = (int)(b >> 44) & 255;
  const unsigned long long f = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  const long long r = (long long)((f * s_log2_c[j]) << 4);    // the 1 drops out
  const long long u = __mul64hi(r, kLog2E_q62);               // r log2(e), 2^-69
  const long long r2 = __mul64hi(r, r);                       // r^2, 2^-78
  const long long t = __mul64hi(r2, kLog2E_q62);              // r^2 log2(e) / 2, 2^-77
  const long long c = __mul64hi(__mul64hi(r2, r), kLog2EThird_q64);  // r^3 log2(e) / 3, 2^-85
  const float rf = (float)(int)(r >> 32) * 0x1p-39f, rf2 = rf * rf;
  const float d = rf2 * rf2 * (0x1p58f * (float)kLog2E) * fmaf(rf, 0.2f, -0.25f);
  return s_log2_q58[j] + (u >> 11) - (t >> 19) + (c >> 27) + (long long)(int)d;
}
// In units of 2^-58 for x in (2^-31, 2^31), and in units of 2^-52 for any positive normal x.
__device__ __forceinline__ long long log2_q58(double x) {
  int e;
  const long long f = log2_parts(x, e);
  return ((long long)e << 58) + f;
}
static __device__ __noinline__ long long log2_q52(double x) {
  int e;
  const long long f = log2_parts(x, e);
  return ((long long)e << 52) + (f >> 6);
}

// x 2^-50 for x in (2^57, 2^63)
__device__ __forceinline__ double q50_to_double(long long x) {
  const int n = __clz((int)(x >> 32));  // 1..6
  const unsigned long long m = ((unsigned long long)x + (1ull << (10 - n))) >> (11 - n);
  return __longlong_as_double(((long long)(1035 - n) << 52) + (long long)m);  // the leading one adds to the exponent
}


// log(x) for positive normal finite x.
__device__ __forceinline__ double log_tab(double x) {
  const long long bits = __double_as_longlong(x);
  const int ex = (int)(bits >> 52) - 1023;
  const long long mb = bits & 0x000fffffffffffffLL;
  const int j = (int)(((mb >> 45) + 1) >> 1);  // nearest 64th of the fraction, 0..64
  const double f = __longlong_as_double(mb | 0x3ff0000000000000LL);
  const double r = fma(f, s_log_inv[j], -1.0);  // |r| <= 1/128
  // log1p(r) = r - r^2/2 + r^3/3 - r^4/4 + r^5/5 - r^6/6 + r^7/7
  double q = fma(r, 1.0 / 7.0, -1.0 / 6.0);
  q = fma(r, q, 1.0 / 5.0);
  q = fma(r, q, -0.25);
  q = fma(r, q, 1.0 / 3.0);
  q = fma(r, q, -0.5);
  const double r2 = r * r;
  const double l1p = fma(r2, q, r);
  // inputs in [0.5, 1): -ln(2 c_j) from the second table, no e ln2 term to cancel against
  if (ex == -1) return s_log_tab_m1[j] + l1p;
  const double e = (double)ex;
  return fma(e, kLn2Hi, s_log_tab[j] + fma(e, kLn2Lo, l1p));
}

// log(x) of the kernels' arguments (temperatures, F_cent, Pr); zero, subnormal, negative, inf
// and NaN inputs fall back to the library log via an integer test of the exponent field.
__device__ __forceinline__ double log_t(double x) {
  const int ef = (int)(__double_as_longlong(x) >> 52);  // sign and biased exponent
  if (ef <= 0 || ef >= 0x7ff) return log(x);
  return log_tab(x);
}

__device__ __forceinline__ double log10_t(double x) { return log_t(x) * kInvLn10; }
__device__ __forceinline__ double exp10_t(double x) { return exp_t(x * kLn10); }

// ---- fp32 <-> fp64 conversions on the integer pipe ----
// On GB300 a cvt between fp32 and fp64 takes an FP64-pipe slot, the same as a DFMA
// (measured), and the mixed-precision right-hand side converts ~50 values per
// evaluation.  These two build the IEEE-754 bit patterns with integer operations
// instead.  Both give a signed zero for magnitudes below the fp32 normal range
// (2^-126) and keep infinities and NaNs.

// fp32 -> fp64: exact for normal numbers
__device__ __forceinline__ double f2d(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t a = u & 0x7fffffffu;
  uint32_t hi = (a >> 3) + 0x38000000u;     // exponent bias 127 -> 1023
  if (a >= 0x7f800000u) hi |= 0x7ff00000u;  // inf / NaN: all-ones exponent
  const bool tiny = a < 0x00800000u;
  hi = tiny ? 0u : hi;
  const uint32_t lo = tiny ? 0u : (u << 29);
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)lo);
}

// fp64 -> fp32, rounded to nearest (ties to even); |d| >= 2^128 gives inf
__device__ __forceinline__ float d2f(double d) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const uint32_t a = hi & 0x7fffffffu;
  uint32_t r = ((a - 0x38000000u) << 3) | (lo >> 29);  // exponent bias 1023 -> 127, 23 bits
  const uint32_t guard = (lo >> 28) & 1u;
  const uint32_t sticky = (lo & 0x0fffffffu) != 0u;
  r += guard & (sticky | (r & 1u));  // a carry out of the fraction bumps the exponent
  r = a >= 0x47f00000u ? 0x7f800000u : r;
  r = (a > 0x7ff00000u || (a == 0x7ff00000u && lo != 0u)) ? 0x7fc00000u : r;
  r = a < 0x38100000u ? 0u : r;
  return __uint_as_float(r | (hi & 0x80000000u));
}

// ---- fp64 reciprocals ----
// An IEEE fp64 divide costs ~9 FP64-pipe slots on GB300 (measured).  Here 1/x starts
// from the hardware approximation rcp.approx.ftz.f64 and takes Newton-Raphson steps
// r <- r + r (1 - x r), each of which squares the relative error (the approximation's
// is near 2^-20): one step for a relative error near 2^-40 (Newton's derivative), two
// for a result within an ulp or two.  x must be finite, nonzero and normal (0 gives
// NaN).
__device__ __forceinline__ double rcp_approx(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  return r;
}
__device__ __forceinline__ double rcp1(double x) {
  const double r = rcp_approx(x);
  return fma(r, fma(-x, r, 1.0), r);
}
__device__ __forceinline__ double rcp2(double x) {
  const double r = rcp1(x);
  return fma(r, fma(-x, r, 1.0), r);
}
// as close as rcp2 in one third-order step, r (1 + d + d^2) with d = 1 - x r: three FP64
// instructions instead of four
__device__ __forceinline__ double rcp3(double x) {
  const double r = rcp_approx(x);
  const double d = fma(-x, r, 1.0);
  return fma(r, fma(d, d, d), r);
}

// ---- fp64 tests and selects on the integer pipe ----
// x positive, finite and normal
__device__ __forceinline__ bool pos_normal(double x) {
  return (uint32_t)__double2hiint(x) - 0x00100000u < 0x7fe00000u;
}
// a >= b for non-negative a, b (the bit patterns of non-negative doubles are ordered)
__device__ __forceinline__ bool ge_nonneg(double a, double b) {
  return __double_as_longlong(a) >= __double_as_longlong(b);
}
// max(|a|, |b|); a NaN operand gives NaN
__device__ __forceinline__ double max_abs(double a, double b) {
  const long long x = __double_as_longlong(a) & 0x7fffffffffffffffLL;
  const long long y = __double_as_longlong(b) & 0x7fffffffffffffffLL;
  return __longlong_as_double(x > y ? x : y);
}
// max(x, 0) (negative values, -0 and NaNs with the sign bit set give +0)
__device__ __forceinline__ double clamp_nonneg(double x) {
  const long long b = __double_as_longlong(x);
  return __longlong_as_double(b & ~(b >> 63));
}

// x = hi + lo for an fp64 x of magnitude below 2^12: hi is x truncated to a multiple of
// 2^-12 (at most 24 significant bits, so exact in fp32) and lo = x - hi (|lo| < 2^-12)
// rounded to fp32, an absolute error below 2^-37.  A signed sum of a few such hi parts
// whose magnitude stays below 2^12 is exact in fp32, so an fp64 sum with heavy
// cancellation (ln K_c from Gibbs functions of magnitude up to a few hundred) is
// assembled in fp32 to within an ulp of the result plus ~1e-11.
// In that range the fraction bits below the grid are an integer of up to 52 bits, whose
// conversion to fp32 rounds as x - hi would: no FP64 instruction.
__device__ __forceinline__ void split_hilo(double x, float &hi, float &lo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  const int n = 1063 - ex;  // fraction bits worth < 2^-12
  if ((unsigned)(n - 29) < 24u) {  // 2^-12 <= |x| < 2^12
    const uint32_t h = (uint32_t)(b >> 32);
    const unsigned long long low = b & ~(~0ull << n), top = b ^ low;
    const uint32_t t = (uint32_t)(top >> 29) - 0xc0000000u;  // exponent bias 1023 -> 127; 24 bits at most, exact
    hi = __uint_as_float((t & 0x7fffffffu) | (h & 0x80000000u));
    const float l = (float)(long long)low * __uint_as_float((uint32_t)(ex - 948) << 23);
    lo = __uint_as_float(__float_as_uint(l) | (h & 0x80000000u));
    return;
  }
  const unsigned long long mask = n >= 53 ? 0ull : (n <= 0 ? ~0ull : (~0ull << n));
  const double h = __longlong_as_double((long long)(b & mask));
  hi = d2f(h);
  lo = d2f(x - h);
}

}  // namespace chem
