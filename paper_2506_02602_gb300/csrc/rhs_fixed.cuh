// rhs_fixed.cuh -- the fp64 right-hand side with everything but its products of concentrations on
// the integer pipe.
//
// An FP64 instruction occupies a warp's sub-partition for 64 cycles on GB300, an integer one for
// 2 and a 32 x 32 -> 64-bit multiply-add for 5, and the fp64 kernel is bound by its FP64
// instructions.  So the temperature solve, the Gibbs functions, the Arrhenius exponents and the
// logarithms are sums of products in 64-bit fixed point (DotQ: 15 cycles a term), which keep more
// digits than fp64 where terms cancel (Gibbs functions of a few hundred have an fp64 rounding
// error of 2^-46, here 2^-50), and the exponentials follow in exp2_q52.
//   - Newton on e(T) evaluates the residual in units down to 2^-40 of e / R_u (fp64 rounds the sums
//     of magnitude 1e6 it has there to 2^-33) and divides it by an fp32 c_v: the step is then off by
//     ~2^-21 of itself, and the iteration goes on until that no longer counts.
//   - Concentrations are per mass (y_k = Y_k / W_k); the powers of rho that belong to the rates
//     enter as log2(rho) in their exponents.
//   - The reverse rate is one exponential of the reaction's Gibbs difference, so a net rate of
//     progress is k_f (prod y_reactants - K prod y_products): 4 FP64 instructions, and reactions
//     of one stoichiometry (duplicates, colliders) share it with their k_f summed.
// A warp's evaluation issued 1040 FP64 instructions in the general form, 637 with only its
// exponentials in fixed point and 300 here; the 1M-cell detonation slice takes 83.2, 49.2 and
// 24.9 ms, a 256-cell batch of 15 steps 3.0, 2.1 and 1.3 ms (one warp's chain of dependent
// instructions).  Integer work now fills the issue slots the FP64 pipe (72 % busy) leaves.
//
// For T in (128, 8192) K, |Y_k| < 1.25, sum |Y_k| <= 1.5, |e| / R_u < 2^26 K mol/kg, rho in
// (2^-64, 2^64) and coefficients within the tables' ranges (MechTables::fixed_ok); anything else takes
// the general form (rhs.cuh).
#pragma once

#include <utility>

#include "fastmath.cuh"
#include "mech.cuh"

namespace chem {

// Per-thread columns, ST threads apart in dynamic shared memory: the advancing solution X, the
// error register E, the stage state U (then the concentrations per mass in its place) and the
// Gibbs functions.  The loops over species stay rolled over them, so their code and their
// coefficients' loads stay few: unrolled, with the columns in registers, a thread wanted 255
// registers (spills at 12 warps an SM) and the code more than the instruction caches.
struct Fp64Cols {
  double *X, *E, *U;
  long long *g;
};
constexpr size_t fp64_cols_bytes(int block) { return (size_t)block * 8 * 4 * NSP; }
template <int ST>
__device__ __forceinline__ Fp64Cols fp64_cols() {
  extern __shared__ double s_cols[];
  Fp64Cols c;
  c.X = s_cols + threadIdx.x;
  c.E = c.X + NSP * ST;
  c.U = c.E + NSP * ST;
  c.g = reinterpret_cast<long long *>(c.U + NSP * ST);
  return c;
}

// Per-block tables of a lane's own NASA-7 range: the energy coefficients in pairs; the Gibbs
// functions' {log2 T, 1/T}, {t, t^2}, {t^3, t^4} and {1, 1/W}.
__shared__ int4 s_qe[2][NSP][3];
__shared__ int4 s_qg[2][NSP][4];

__device__ __forceinline__ int4 pack_q(const QCoef &a, const QCoef &b) { return make_int4(a.h, a.l, b.h, b.l); }
// solve_T_fixed's table
__device__ __forceinline__ void load_energy_table(const MechTables &mt) {
  for (int i = threadIdx.x; i < 2 * NSP; i += blockDim.x) {
    const int r = i / NSP, k = i % NSP;
    for (int j = 0; j < 3; ++j) s_qe[r][k][j] = pack_q(mt.qe[r][k][2 * j], mt.qe[r][k][2 * j + 1]);
  }
  __syncthreads();
}
__device__ __forceinline__ void load_fixed_tables(const MechTables &mt) {
  load_exp2_tables();
  load_log2_table();
  load_energy_table(mt);
  for (int i = threadIdx.x; i < 2 * NSP; i += blockDim.x) {
    const int r = i / NSP, k = i % NSP;
    s_qg[r][k][0] = pack_q(mt.qg[r][k][0], mt.qg[r][k][1]);
    s_qg[r][k][1] = pack_q(mt.qgt[r][k][0], mt.qgt[r][k][1]);
    s_qg[r][k][2] = pack_q(mt.qgt[r][k][2], mt.qgt[r][k][3]);
    const long long w = __double_as_longlong(mt.invW[k]);
    s_qg[r][k][3] = make_int4((int)(mt.qg1[r][k] >> 32), (int)mt.qg1[r][k], (int)(w >> 32), (int)w);
  }
  __syncthreads();
}

constexpr int kRoll = 3;  // species of a rolled loop's step

// 128 < T < 8191.996 and 2^-64 < rho < 2^64, on the high words
__device__ __forceinline__ bool fixed_T(double T) {
  return (uint32_t)__double2hiint(T) - 0x40600001u < 0x40bfffffu - 0x40600001u;
}
__device__ __forceinline__ bool fixed_rho(double rho) {
  return (uint32_t)__double2hiint(rho) - 0x3bf00000u < 0x43f00000u - 0x3bf00000u;
}

// Temperature from (e, Y) as solve_T: the same iteration from the same guess.  False when an
// argument is out of range or an iterate leaves it, or without convergence; T is then unchanged.
//
// The residual is in units of 2^-q_res of e/R_u (2^-36 below T_mid and 2^-35 above for the mechanisms
// here).  Sums are rounded and the limbs centred, so that what is dropped does not add up, and where
// the residual is small (2^9 at most) its last multiplication and its constant term keep 4 more bits,
// modulo 2^64.  So T is within 7e-16 of the root (rms 1e-16 to 1.6e-16), as in
// fp64; with units of 2^-33 and everything truncated it was off by up to 4e-14 (rms 1e-15 to 1e-14).
// The step's fp32 slope leaves 2^-21 of it; a step of 4e-10 T ends the iteration.
template <int ST>
__device__ __forceinline__ bool solve_T_fixed(const MechTables &mt, const double *U, double eR, double &T) {
  constexpr int kFine = 4;
  const uint32_t eh = (uint32_t)__double2hiint(eR) & 0x7fffffffu;
  if (!fixed_T(T) || eh >= 0x41900000u) return false;  // |eR| < 2^26
  long long Tq = (long long)abs_q<50>(T);
  long long m[6];
  unsigned long long m5f = 0;
  float d[5];
  int range = -1, shift = 0;
  float unit = 0.0f;
  bool done = false;
  for (int it = 0; it < 30; ++it) {
    const int r = Tq >= mt.qT_mid;
    if (r != range) {  // mixture coefficients
      range = r;
      shift = 13 - mt.q_log2[r];
      unit = __int_as_float((127 + 13 - shift) << 23);
      DotQ<1> s[6];
#pragma unroll
      for (int i = 0; i < 6; ++i) s[i] = {0, i < 5 ? 1ll << 30 : 0};  // halves: the values are rounded
      uint32_t big = 0, sum = 0;
#pragma unroll kRoll
      for (int k = 0; k < NSP; ++k) {
        const double yk = U[k * ST];
        big = max(big, (uint32_t)__double2hiint(yk) & 0x7fffffffu);
        const long long sy = (long long)__double2hiint(yk) >> 31;
        const long long ay = (long long)abs_q<62>(yk);
        sum += (uint32_t)(ay >> 36);
        const Limbs<1> y = limbs_centred<1>((ay ^ sy) - sy);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const int4 q = s_qe[r][k][i];
          s[2 * i].add(q.x, q.y, y);
          s[2 * i + 1].add(q.z, q.w, y);
        }
      }
      if (big >= 0x3ff40000u || sum > 0x06000000u - NSP) break;  // |Y| < 1.25, sum |Y| <= 1.5
#pragma unroll
      for (int i = 0; i < 6; ++i) m[i] = s[i].value();
      m5f = s[5].template fine<kFine>();
      {  // e/R_u, truncated
        const int n = (int)(eh >> 20) - 1075 + mt.q_res[r];
        const unsigned long long a =
            ((unsigned long long)__double_as_longlong(eR) & 0x000fffffffffffffull) | 0x0010000000000000ull;
        const unsigned long long c = n >= 0 ? a << n : a >> min(-n, 63);
        const unsigned long long f = n + kFine >= 0 ? a << (n + kFine) : a >> min(-n - kFine, 63);
        const bool neg = __double2hiint(eR) < 0;
        m[5] -= neg ? -(long long)c : (long long)c;
        m5f -= neg ? 0ull - f : f;
      }
#pragma unroll
      for (int i = 0; i < 5; ++i) d[i] = (float)(i + 1) * __ll2float_rn(m[i]);
    }
    const long long t = Tq << shift;
    const Limbs<1> tl = limbs_centred<1>(t);
    long long e = m[4];
#pragma unroll
    for (int i = 3; i >= 0; --i) e = MulQ(e, tl).value() + m[i];
    const MulQ p(e, tl);
    e = p.value() + m[5];
    const bool fine = (uint32_t)(int)(e >> 32) + 0x1000u < 0x2000u;  // |e| < 2^44: a few K at most
    if (fine) e = (long long)(p.template fine<kFine>() + m5f);
    const float tf = __ll2float_rn(t) * 0x1p-63f;
    const float cv = fmaf(tf, fmaf(tf, fmaf(tf, fmaf(tf, d[4], d[3]), d[2]), d[1]), d[0]);
    const float dT = __fdividef(__ll2float_rn(e), cv) * (fine ? unit * (1.0f / (1 << kFine)) : unit);
    if (!(fabsf(dT) < 4096.0f)) break;
    Tq -= __float2ll_rn(dT * 0x1p50f);
    if ((uint32_t)(Tq >> 32) - 0x02000001u >= 0x7fffffffu - 0x02000001u) break;
    const float Tf = (float)(int)(Tq >> 32) * 0x1p-18f;
    done = fine && fabsf(dT) <= 4e-10f * Tf;
    if (done) break;
  }
  if (done) T = q50_to_double(Tq);
  return done;
}

struct RateInputsQ {
  double T, invT, ctot;
  Limbs<2> lT, iT;       // log2 T (Q58), 1/T (Q70)
  long long lrho, lRT;   // log2 rho (Q52), log2(rho R_u T / p_ref) (Q50)
  const double *U;       // column of Y_k / W_k, clamped
  double y[NSP];         // the same
  long long g[NSP];      // -g_k / (R_u T ln2) (Q50)
};

// log2 x; zero, negative, subnormal and non-finite arguments by the library
__device__ __forceinline__ double log2_any(double x) {
  if (pos_normal(x)) return (double)log2_q52(x) * 0x1p-52;
  return log(x) * kLog2E;
}

// log2 of A T^b exp(-Ta / T) times rho^kPow, Q52
template <int kPow>
__device__ __forceinline__ long long rate_log2(int64_t a, const QCoef &b, const QCoef &h, const RateInputsQ &in) {
  DotQ<2> s{a + kPow * in.lrho, 0};
  s.add(b.h, b.l, in.lT);
  s.add(h.h, h.l, in.iT);
  return s.value();
}

// Third-body sums [M] / rho go through the list of efficiencies that differ from the base, 1 or 0,
// a rolled loop of a few entries: unrolled over all species under their mask, the compiler
// computed every term and selected, 41 FP64 instructions a warp more.
// Forward rate coefficient of reaction J times rho^(order - 1), third body and fall-off included:
// in the units of y.  With kK also K = 2^lK, whose exponential joins one of the rate's.
template <int ST, int J, bool kK>
__device__ __forceinline__ double rate_fixed(const MechTables &mt, const RateInputsQ &in, long long lK, double &K) {
  constexpr RxStruct R = kRx[J];
  constexpr int pw = n_reac(R) - 1;
  double M = 0.0;
  if constexpr (R.type != ELEM) {
    M = mt.m_base[J] ? in.ctot : 0.0;
#pragma unroll 1
    for (int i = 0; i < mt.m_n[J]; ++i) M = fma(mt.m_c[J][i], in.U[mt.m_k[J][i] * ST], M);
  }
  if constexpr (R.type != FALLOFF) {
    const long long l = limit_q<52>(rate_log2<pw + (R.type == THIRD_BODY)>(mt.qA[J], mt.qB[J], mt.qH[J], in));
    double kf;
    if constexpr (kK) {
      const double2 v = exp2_q52(l, lK);
      kf = v.x;
      K = v.y;
    } else {
      kf = exp2_q52(l);
    }
    return R.type == THIRD_BODY ? kf * M : kf;
  } else {
    const long long li = rate_log2<pw>(mt.qA[J], mt.qB[J], mt.qH[J], in);
    const long long l0 = rate_log2<pw + 1>(mt.qA0[J], mt.qB0[J], mt.qH0[J], in);
    const double2 v = exp2_q52(limit_q<52>(li), limit_q<52>(l0));
    const double k0M = v.y * M;
    // k_inf Pr / (1 + Pr), Pr = k0 M / k_inf
    double kf = k0M > 0.0 ? v.x * (k0M * rcp3(v.x + k0M)) : 0.0;
    if constexpr (R.troe_n != 0) {
      // Troe broadening (Gilbert, Luther & Troe 1983) in log2: with x = lg Pr - 0.4 - 0.67 lg Fc and
      // d = 0.75 - 1.27 lg Fc - 0.14 x, log F = log Fc d^2 / (d^2 + x^2)
      const double a = mt.troe_a[J];
      const double2 f = exp2_q52(to_q52(-in.T * mt.troe_q3[J]), to_q52(-in.T * mt.troe_q1[J]));
      double Fc = fma(a, f.y, (1.0 - a) * f.x);
      if constexpr (R.troe_n == 4) {
        const double2 w = exp2_q52(to_q52(-mt.troe_q2[J] * in.invT), lK);
        Fc += w.x;
        K = w.y;
      }
      const double lFc = log2_any(Fc);
      const double lPr = fma((double)((l0 >> 2) - (li >> 2)), 0x1p-50, log2_any(M));
      const double x = fma(-0.67, lFc, lPr - 0.4 * kLog2_10);
      const double d = fma(-0.14, x, fma(-1.27, lFc, 0.75 * kLog2_10));
      const double d2 = d * d;
      const double f2 = lFc * (d2 * rcp3(fma(x, x, d2)));
      const long long lF = to_q52(f2);
      double F;
      if constexpr (kK && R.troe_n != 4) {
        const double2 w = exp2_q52(lF, lK);
        F = w.x;
        K = w.y;
      } else {
        F = exp2_q52(lF);
      }
      // Without third bodies log Pr is infinite and the rate zero.  Else a factor that is no number
      // (F_cent zero, negative or NaN) makes the rate none, as in the general form: to_q52 has none.
      kf = k0M > 0.0 ? kf * (is_nan(f2) ? f2 : F) : 0.0;
    } else if constexpr (kK) {
      K = exp2_q52(lK);
    }
    return kf;
  }
}

__host__ __device__ constexpr bool same_species(int a0, int a1, int b0, int b1) {
  return (a0 == b0 && a1 == b1) || (a0 == b1 && a1 == b0);
}
// the first reaction of J's stoichiometry
__host__ __device__ constexpr int rx_leader(int j) {
  for (int i = 0; i < j; ++i)
    if (same_species(kRx[i].r0, kRx[i].r1, kRx[j].r0, kRx[j].r1) &&
        same_species(kRx[i].p0, kRx[i].p1, kRx[j].p0, kRx[j].p1))
      return i;
  return j;
}
__host__ __device__ constexpr int rx_group(int j) {
  int n = 0;
  for (int i = 0; i < NRX; ++i) n += rx_leader(i) == j;
  return n;
}
// whether a reaction before J changes species k
__host__ __device__ constexpr bool rx_touched(int k, int j) {
  for (int i = 0; i < j; ++i)
    if (kRx[i].r0 == k || kRx[i].r1 == k || kRx[i].p0 == k || kRx[i].p1 == k) return true;
  return false;
}

// bit k: some reaction changes species k
__host__ __device__ constexpr uint32_t rx_reactive() {
  uint32_t m = 0;
  for (int k = 0; k < NSP; ++k) m |= (uint32_t)rx_touched(k, NRX) << k;
  return m;
}
constexpr uint32_t kReactive = rx_reactive();

// wdot_k +-= nu q: an assignment where it is the species' first term
template <int J, int K, int NU>
__device__ __forceinline__ void rate_add(double q, double (&wdot)[NSP]) {
  if constexpr (!rx_touched(K, J)) wdot[K] = NU * q;
  else if constexpr (NU == 1) wdot[K] += q;
  else if constexpr (NU == -1) wdot[K] -= q;
  else wdot[K] = fma((double)NU, q, wdot[K]);
}

template <int ST, int J, int I>
__device__ __forceinline__ void rate_member(const MechTables &mt, const RateInputsQ &in, double &kF, double &kR) {
  if constexpr (I != J && rx_leader(I) == J) {
    double none;
    const double k = rate_fixed<ST, I, false>(mt, in, 0, none);
    kF += k;
    if (mt.reversible[I]) kR += k;
  }
}

// Net rate of progress of the reactions of J's stoichiometry into wdot, J the first of them
template <int ST, int J, int... I>
__device__ __forceinline__ void reaction_fixed(const MechTables &mt, const RateInputsQ &in, double (&wdot)[NSP],
                                               std::integer_sequence<int, I...>) {
  if constexpr (rx_leader(J) == J) {
    constexpr RxStruct R = kRx[J];
    constexpr int dnu = n_prod(R) - n_reac(R);
    static_assert(dnu >= -1 && dnu <= 1, "compiled structure assumes |sum nu| <= 1");
    long long l = in.g[R.r0] - in.g[R.p0] + dnu * in.lRT;
    if constexpr (R.r1 >= 0) l += in.g[R.r1];
    if constexpr (R.p1 >= 0) l -= in.g[R.p1];
    double K;
    double kF = rate_fixed<ST, J, true>(mt, in, limit_q<50>(l) << 2, K);
    double yr = in.y[R.r0], yp = in.y[R.p0];
    if constexpr (R.r1 >= 0) yr *= in.y[R.r1];
    if constexpr (R.p1 >= 0) yp *= in.y[R.p1];
    double q;
    if constexpr (rx_group(J) > 1) {
      double kR = mt.reversible[J] ? kF : 0.0;
      (rate_member<ST, J, I>(mt, in, kF, kR), ...);
      q = fma(kF, yr, -(kR * (K * yp)));
    } else {
      q = kF * (mt.reversible[J] ? fma(-K, yp, yr) : yr);
    }
    if constexpr (R.r0 == R.r1) {
      rate_add<J, R.r0, -2>(q, wdot);
    } else {
      rate_add<J, R.r0, -1>(q, wdot);
      if constexpr (R.r1 >= 0) rate_add<J, R.r1, -1>(q, wdot);
    }
    if constexpr (R.p0 == R.p1) {
      rate_add<J, R.p0, 2>(q, wdot);
    } else {
      rate_add<J, R.p0, 1>(q, wdot);
      if constexpr (R.p1 >= 0) rate_add<J, R.p1, 1>(q, wdot);
    }
  }
}

template <int ST, int... J>
__device__ __forceinline__ void all_reactions_fixed(const MechTables &mt, const RateInputsQ &in, double (&wdot)[NSP],
                                                    std::integer_sequence<int, J...> seq) {
  (reaction_fixed<ST, J>(mt, in, wdot, seq), ...);
}

// dY/dt at T from solve_T_fixed; U becomes the concentrations per mass.
template <int ST>
__device__ __forceinline__ void rates_fixed(const MechTables &mt, const Fp64Cols &m, double rho, double T,
                                            double (&F)[NSP]) {
  RateInputsQ in;
  in.U = m.U;
  in.T = T;
  in.invT = rcp3(T);
  const long long lT = log2_q58(T);
  in.lT = limbs<2>(lT);
  in.iT = limbs<2>((long long)abs_q<70>(in.invT));
  in.lrho = log2_q52(rho);
  in.lRT = (lT >> 8) + mt.qRP + (in.lrho >> 2);
  {
    const int range = ge_nonneg(T, mt.T_mid);
    const long long t1 = (long long)abs_q<50>(T) << (13 - mt.q_log2[range]);
    const long long t2 = mul_q63(t1, t1);
    const Limbs<4> t[4] = {limbs<4>(t1), limbs<4>(t2), limbs<4>(mul_q63(t2, t1)), limbs<4>(mul_q63(t2, t2))};
    in.ctot = 0.0;
#pragma unroll kRoll
    for (int k = 0; k < NSP; ++k) {
      const int4 q = s_qg[range][k][0], q1 = s_qg[range][k][1], q2 = s_qg[range][k][2], q3 = s_qg[range][k][3];
      DotQ<2> a{(long long)(((unsigned long long)(uint32_t)q3.x << 32) | (uint32_t)q3.y), 0};
      a.add(q.x, q.y, in.lT);
      a.add(q.z, q.w, in.iT);
      DotQ<4> b{0, 0};
      b.add(q1.x, q1.y, t[0]);
      b.add(q1.z, q1.w, t[1]);
      b.add(q2.x, q2.y, t[2]);
      b.add(q2.z, q2.w, t[3]);
      m.g[k * ST] = a.value() + (b.value() >> 6);
      const double y = clamp_nonneg(m.U[k * ST] * __hiloint2double(q3.z, q3.w));
      m.U[k * ST] = y;
      in.ctot += y;
    }
  }
#pragma unroll
  for (int k = 0; k < NSP; ++k) {
    in.y[k] = m.U[k * ST];
    in.g[k] = m.g[k * ST];
  }
  double wdot[NSP];
  all_reactions_fixed<ST>(mt, in, wdot, std::make_integer_sequence<int, NRX>{});
#pragma unroll
  for (int k = 0; k < NSP; ++k) F[k] = ((kReactive >> k) & 1) ? wdot[k] * mt.W[k] : 0.0;
}

}  // namespace chem
